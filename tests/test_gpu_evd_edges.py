"""Block Jacobi at the edges of its blocks (16 columns, pairs of 32, chunks of 640) and on covariances without full rank:
dead features, repeated features, fewer samples than features, none at all."""
import numpy as np
import pytest

from fwtest_util import TOL_FP32, rel_fro, t2n
from test_gpu_evd import oracle_state, scratch_for, spd32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2010_01546_b200 import binding as B, build
    build.build_library()
    return torch, B


def whiten(env, Phi32, g_max):
    torch, B = env
    M = Phi32.shape[0]
    L = B.Layer(M, 4, beta=0.0, gamma=1.0)
    L.set(B.FW_F_PHIX, torch.from_numpy(Phi32).cuda())
    scratch, nb = scratch_for(torch, B, M)
    B.fw_evd_whiten(L.handle, scratch, nb, g_max)
    assert L.sync_status() == B.FW_OK
    To, Qo, _, _ = oracle_state(Phi32, L.desc.eps, g_max if g_max > 0 else None)
    T, Q = t2n(L.get(B.FW_F_T)).reshape(M, M), t2n(L.get(B.FW_F_Q)).reshape(M, M)
    assert rel_fro(T, To) <= TOL_FP32 and rel_fro(Q, Qo) <= TOL_FP32
    assert np.array_equal(T, T.T) and np.array_equal(Q, Q.T)


@pytest.mark.parametrize("M", [15, 16, 17, 31, 32, 33, 48, 129, 640, 641])
def test_block_edges(env, M):
    whiten(env, spd32(M, 1e2, 300 + M), 0.0)
    whiten(env, spd32(M, 1e2, 300 + M), 3.0)


@pytest.mark.parametrize("kind", ["dead", "repeated", "few_samples", "zero", "diagonal"])
def test_no_full_rank(env, kind):
    rng = np.random.default_rng(11)
    M = 70
    X = rng.standard_normal((400 if kind != "few_samples" else 20, M))
    if kind == "dead":
        X[:, [3, 16, 17, 69]] = 0.0
    if kind == "repeated":
        X[:, 40:44] = X[:, [5]]
    Phi = (X.T @ X / X.shape[0]).astype(np.float32)
    if kind == "zero":
        Phi[:] = 0.0
    if kind == "diagonal":
        Phi = np.diag(np.logspace(0, -3, M)).astype(np.float32)
    Phi = np.triu(Phi) + np.triu(Phi, 1).T
    for g_max in ((0.0, 10.0) if kind != "zero" else (0.0,)):
        whiten(env, Phi, g_max)


def test_eigenvalues_not_told_from_zero(env):
    """Up to 1e-13 of the largest eigenvalue the gain is that of zero, 1 / eps (Eq. 10), whatever eps; above, 1 / lambda."""
    torch, B = env
    M = 40
    lam = np.logspace(0, -11, M)
    lam[[7, 33]] = 1e-12, 1e-15
    L = B.Layer(M, 4, beta=0.0, gamma=1.0, eps=1e-18)
    L.set(B.FW_F_PHIX, torch.from_numpy(np.diag(lam).astype(np.float32)).cuda())
    scratch, nb = scratch_for(torch, B, M)
    B.fw_evd_whiten(L.handle, scratch, nb, 0.0)
    want = 1.0 / np.sqrt(lam)
    want[33] = 1e9
    T = t2n(L.get(B.FW_F_T))
    assert np.abs(np.diag(T) / want - 1.0).max() <= TOL_FP32 and np.abs(T - np.diag(np.diag(T))).max() == 0.0
    assert L.sync_status() == B.FW_OK
