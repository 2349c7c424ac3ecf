"""The gradient transform of several small tensor-core layers in one call: sets on both sides of the rule that picks the kernel, layers
whose K takes fewer CTAs than the cluster they are given, more layers than a launch holds."""
import numpy as np
import pytest

from fwtest_util import t2n

pytestmark = pytest.mark.gpu

# (N, M) of the layers and the launches of the call, the bias step's included: one for sixteen layers by the kernel of small products; by CTA pairs
# another where K is split
SETS = [([(10, 1000)] * 3, 2), ([(1, 1000)] * 4, 2), ([(1, 1000)] * 8, None), ([(1, 1000)] * 37, None), ([(10, 576)] * 6, 2),
        ([(10, 576)] * 12, None), ([(1, 300)] * 20, 3), ([(10, 1000)] + [(16, 144)] * 15, 3),
        ([(10, 1000), (32, 576), (32, 300), (32, 64)], 2), ([(64, 300)] * 3 + [(32, 144)] * 3 + [(16, 576)] * 2, 2),
        ([(1, 1000)] + [(16, 64)] * 8, 2), ([(5, 20)] * 17 + [(3, 340)], 3)]


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2010_01546_b200 import binding as B, build
    build.build_library()
    return torch, B


@pytest.mark.parametrize("layers,launches", SETS)
def test_groups(env, layers, launches):
    """Both operands lose up to 2^-10 of a value to TF32 and a chain of M additions at most 2^-22 an addition."""
    torch, B = env
    rng = np.random.default_rng(len(layers))
    cu = lambda a: torch.from_numpy(a).cuda()
    Ls, Qs = [], {}
    for k, (N, M) in enumerate(layers):
        L = B.Layer(M, N, beta=0.0, gamma=1.0, prec=B.FW_PREC_TF32)
        if M not in Qs:
            T = (np.eye(M) + 0.3 * rng.standard_normal((M, M)) / np.sqrt(M)).astype(np.float32)
            Qs[M] = cu(T)
        L.set(B.FW_F_T, Qs[M])
        Ls.append(L)
    G = [rng.standard_normal((N, M)).astype(np.float32) for N, M in layers]
    W = [torch.zeros(N, M, device="cuda") for N, M in layers]
    zero = [torch.zeros(N, device="cuda") for N, _ in layers]
    Gd = [cu(g) for g in G]
    n0 = B.fw_launch_count()
    B.fw_group_grad_transform_step([L.handle for L in Ls], Gd, W, zero, zero, 1.0)
    assert launches is None or B.fw_launch_count() - n0 == launches
    for L, g, w, (N, M) in zip(Ls, G, W, layers):
        Q = t2n(L.get(B.FW_F_QS)).reshape(M, M).astype(np.float64)
        tol = (2.05 * 2.0 ** -10 + M * 2.0 ** -22) * (np.abs(g).astype(np.float64) @ np.abs(Q))
        assert np.all(np.abs(t2n(w) + g.astype(np.float64) @ Q) <= tol)
        assert L.sync_status() == B.FW_OK
