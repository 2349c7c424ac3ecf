"""Re-sync products Phi_y = T Phi_x T^T of the tensor-core engine at the edges of their tiles and boxes, with and without
leakage, from every origin of T: set, reduced (on chip and by a team of CTAs), from the eigenvalues, reset."""
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


def check(L, B, Phi):
    """Four operands are rounded to TF32 (2^-11 each) and each of the two chains of M additions loses at most 2^-22 an addition."""
    M = Phi.shape[0]
    T = t2n(L.get(B.FW_F_T)).reshape(M, M).astype(np.float64)
    Y = t2n(L.get(B.FW_F_PHIY)).reshape(M, M)
    Phi = Phi.astype(np.float64)
    scale = np.abs(T) @ np.abs(Phi) @ np.abs(T).T
    assert np.all(np.abs(Y - T @ Phi @ T.T) <= (4.1 * 2.0 ** -11 + 2 * M * 2.0 ** -22) * scale)
    assert np.array_equal(Y, Y.T)
    assert L.sync_status() == B.FW_OK


@pytest.mark.parametrize("gamma", [1.0, 0.99])
@pytest.mark.parametrize("M", [16, 20, 60, 96, 100, 128, 132, 260, 272, 640, 1020, 1024, 1028, 1100, 1344, 1540])
def test_resync_after_every_origin_of_T(env, M, gamma):
    torch, B = env
    rng = np.random.default_rng(M)
    cu = lambda a: torch.from_numpy(a).cuda()
    L = B.Layer(M, 4, beta=0.0, gamma=gamma, prec=B.FW_PREC_TF32)
    P0, P1 = phi(rng, M), phi(rng, M)
    T = (np.eye(M) + 0.3 * rng.standard_normal((M, M)) / np.sqrt(M)).astype(np.float32)
    L.set(B.FW_F_T, cu(T))
    L.set(B.FW_F_PHIX, cu(P0))
    L.cond_reduce(0, 0)
    check(L, B, P0)                                   # a T that was set
    L.cond_reduce(2, 3)
    L.set(B.FW_F_PHIX, cu(P1))
    L.cond_reduce(0, 0)
    check(L, B, P1)                                   # that two steps changed
    if M <= 300:
        n = B.fw_evd_scratch_bytes(M)
        scratch = torch.empty((n + 255) // 256 * 256, dtype=torch.uint8, device="cuda")
        B.fw_group_evd_whiten([L.handle], [scratch], [n], 10.0)
        L.set(B.FW_F_PHIX, cu(P0))
        L.cond_reduce(0, 0)
        check(L, B, P0)                               # from the eigenvalues of P1
    B.fw_layer_reset(L.handle)
    L.set(B.FW_F_PHIX, cu(P0))
    L.cond_reduce(2, 3)                               # from T = I
    L.set(B.FW_F_PHIX, cu(P1))
    L.cond_reduce(0, 0)
    check(L, B, P1)
