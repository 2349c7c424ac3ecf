"""Calls of more steps than T and Q take together, on chip: the bits of the same steps in several calls, and one launch for layers of
one CTA each."""
import numpy as np
import pytest

from fwtest_util import t2n

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2010_01546_b200 import binding as B, build
    build.build_library()
    return torch, B


def phi(rng, M):
    A = rng.standard_normal((M, M + 8)) / np.sqrt(M)
    P = (A @ A.T).astype(np.float32)
    return np.triu(P) + np.triu(P, 1).T


@pytest.mark.parametrize("prec", ["fp32", "tf32"])
@pytest.mark.parametrize("sizes", [[1], [33], [64], [65], [130], [256], [576], [623], [16, 40, 64], [16, 64, 100, 300], [144] * 9])
def test_the_same_bits(env, sizes, prec):
    torch, B = env
    rng = np.random.default_rng(sum(sizes))
    mats = [torch.from_numpy(phi(rng, M)).cuda() for M in sizes]
    fields = (B.FW_F_T, B.FW_F_Q, B.FW_F_PHIY)

    def fresh(beta):
        Ls = [B.Layer(M, 2, beta=beta, gamma=1.0, prec=B.FW_PREC_FP32 if prec == "fp32" else B.FW_PREC_TF32) for M in sizes]
        for L, P in zip(Ls, mats):
            assert B.fw_recursion_on_chip(L.desc)
            L.set(B.FW_F_PHIX, P)
        B.fw_group_cond_reduce([L.handle for L in Ls], 0, 0)
        return Ls

    def run(Ls, K, traces):
        n0 = B.fw_launch_count()
        B.fw_group_cond_reduce([L.handle for L in Ls], K, 3, traces)
        return B.fw_launch_count() - n0

    whole, parts, smooth = fresh(0.0), fresh(0.0), fresh(0.25)
    tr = [torch.zeros(27, 4, device="cuda") for _ in sizes]
    ts = [torch.zeros(27, 4, device="cuda") for _ in sizes]
    n = run(whole, 27, tr)
    assert n == 1 if max(sizes) <= 64 else n > 1
    k = 0
    for step in (8, 3, 1, 15):
        run(parts, step, [t[k:] for t in ts])
        k += step
    run(smooth, 27, tr)
    for i, M in enumerate(sizes):
        assert torch.equal(tr[i], ts[i])
        for f in fields:
            assert torch.equal(whole[i].get(f), parts[i].get(f))
            assert torch.equal(whole[i].get(f), smooth[i].get(f))
        # Qs starts at I and is smoothed once a call: two roundings of sums of at most |I| + |Q|
        Q, Qs = (t2n(smooth[i].get(f)).astype(np.float64).reshape(M, M) for f in (B.FW_F_Q, B.FW_F_QS))
        assert np.all(np.abs(Qs - (0.25 * np.eye(M) + 0.75 * Q)) <= 2.0 ** -22 * (np.eye(M) + np.abs(Q)))
        for L in (whole[i], parts[i], smooth[i]):
            assert L.sync_status() in (B.FW_OK, B.FW_WARN_NO_SUBSPACE)
