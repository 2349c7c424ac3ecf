"""Covariance updates one right after the other on the same workspaces, with other data each time: the bits of the same updates with
the device waited for in between."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2010_01546_b200 import binding as B, build
    build.build_library()
    return torch, B


@pytest.mark.parametrize("prec", ["fp32", "tf32"])
@pytest.mark.parametrize("sizes", [[(1, 7)], [(64, 128)], [(75, 901)], [(96, 20000)], [(147, 3000)], [(402, 1500)], [(580, 900)],
                                   [(27, 4000), (147, 600), (64, 300)], [(1000, 300), (33, 5000)]])
def test_updates_in_a_row(env, sizes, prec):
    torch, B = env
    g = torch.Generator(device="cuda").manual_seed(1)
    calls = 40
    X = [[torch.rand(r, M, generator=g, device="cuda") for M, r in sizes] for _ in range(4)]
    rows, ld = [r for _, r in sizes], [M for M, _ in sizes]

    def run(wait):
        Ls = [B.Layer(M, 2, alpha=0.5, beta=0.0, gamma=1.0, prec=B.FW_PREC_FP32 if prec == "fp32" else B.FW_PREC_TF32) for M in ld]
        hs, out = [L.handle for L in Ls], []
        for k in range(calls):
            if k % 10 == 9:                       # a block over two calls now and then
                B.fw_group_cov_update(hs, X[0], rows, ld, B.FW_COV_ACCUMULATE)
            B.fw_group_cov_update(hs, X[k % 4], rows, ld)
            if wait:
                torch.cuda.synchronize()
            if k % 4 == 3:
                out += [L.get(f) for L in Ls for f in (B.FW_F_PHIX, B.FW_F_MU, B.FW_F_PHI_DIAG)]
        assert all(L.sync_status() == B.FW_OK for L in Ls)
        return out

    for a, b in zip(run(False), run(True)):
        assert torch.equal(a, b)
