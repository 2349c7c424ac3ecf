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


@pytest.mark.parametrize("M", [16, 47, 640])
@pytest.mark.parametrize("kind", ["graded", "singular", "indefinite", "clustered"])
def test_start_from_the_factor_or_from_phi(env, M, kind):
    """Graded matrices (D A D, D powers of two: eigenvalues over eight decades) are factored; one exact dependence, or a
    negative eigenvalue, and the rotations start from Phi itself.  Clustered: eigenvalues that differ by less than fp32 can
    tell."""
    rng = np.random.default_rng(M)
    B = rng.standard_normal((M, 2 * M)) / np.sqrt(2 * M)
    Phi = (B @ B.T).astype(np.float32).astype(np.float64)
    if kind == "graded":
        d = 2.0 ** -np.round(np.linspace(0, 13, M))
        Phi = d[:, None] * Phi * d[None, :]
    elif kind == "singular":
        Phi[:, -1] = Phi[:, 0]
        Phi[-1, :] = Phi[0, :]
        Phi[-1, -1] = Phi[0, 0]
    elif kind == "clustered":
        q, _ = np.linalg.qr(rng.standard_normal((M, M)))
        Phi = (q * (1.0 + 1e-7 * rng.standard_normal(M) + (np.arange(M) < M // 4))) @ q.T
    else:
        Phi[M // 2, M // 2] -= 2.0
    Phi = np.triu(Phi) + np.triu(Phi, 1).T
    whiten(env, Phi.astype(np.float32), 3.0)


def test_few_ctas_per_long_layer(env):
    """64 layers of 42 block rows in two chunks each: two CTAs a layer, so more of its own block rows than are updated per
    staging."""
    torch, B = env
    M, n = 657, 64
    Phis = [spd32(M, 1e2, 40 + i) for i in range(2)]
    Ls, scr = [], []
    for i in range(n):
        L = B.Layer(M, 4, beta=0.0, gamma=1.0)
        L.set(B.FW_F_PHIX, torch.from_numpy(Phis[i % 2]).cuda())
        Ls.append(L); scr.append(scratch_for(torch, B, M))
    B.fw_group_evd_whiten([L.handle for L in Ls], [s[0] for s in scr], [s[1] for s in scr], 0.0)
    for i in (0, 1, n - 2, n - 1):
        assert Ls[i].sync_status() == B.FW_OK
        To, Qo, _, _ = oracle_state(Phis[i % 2], Ls[i].desc.eps, None)
        assert rel_fro(t2n(Ls[i].get(B.FW_F_T)), To) <= TOL_FP32 and rel_fro(t2n(Ls[i].get(B.FW_F_Q)), Qo) <= TOL_FP32


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


def rounds_taken(torch, scratch, M):
    """Rounds of the last call: the scratch starts with the barrier words, each CTA's count of barriers, one after loading, one per
    16 rows of the factor and one more, then one a round."""
    return (int(scratch[:1024].view(torch.int32)[64]) >> 16) - 1 - ((M + 15) // 16 + 1)


# (a, b, d) of fp32 blocks [[a, b], [b, d]]: b / a, the cosine of their factor's two columns, exceeds the rotations' tolerance of
# 1e-14 by a part in 1e7, less than fp32 products tell
BARELY = [("0x1.4471060000000p+1", "0x1.c89c620000000p-46", "0x1.a3703c0000000p+1"),
          ("0x1.94766e0000000p+0", "0x1.1c9d840000000p-46", "0x1.4c46580000000p+1"),
          ("0x1.ef237e0000000p+1", "0x1.5c6c420000000p-45", "0x1.1e0fb00000000p+0")]


@pytest.mark.parametrize("abd", BARELY)
@pytest.mark.parametrize("M,j", [(2, 1), (34, 33)])
def test_rounds_end_with_a_pair_at_the_tolerance(env, M, j, abd):
    """A pair whose cosine lies at the tolerance counts as rotated only where it is rotated: otherwise it is found again in every
    sweep, up to the last one allowed.  In a visit of all pairs (M = 2) and of blocks 0 and 2 (M = 34)."""
    torch, B = env
    a, b, d = (float.fromhex(x) for x in abd)
    assert 1e-14 < b / a < 1e-14 * (1 + 1.3e-7)
    Phi = np.diag(np.linspace(1.0, 3.0, M)).astype(np.float32)
    Phi[0, 0], Phi[j, j], Phi[0, j], Phi[j, 0] = a, d, b, b
    L = B.Layer(M, 4, beta=0.0, gamma=1.0)
    L.set(B.FW_F_PHIX, torch.from_numpy(Phi).cuda())
    scratch, nb = scratch_for(torch, B, M)
    B.fw_evd_whiten(L.handle, scratch, nb, 0.0)
    assert L.sync_status() == B.FW_OK
    assert 1 <= rounds_taken(torch, scratch, M) <= 3 * ((((M + 15) // 16 + 1) & ~1) - 1)
    T = t2n(L.get(B.FW_F_T)).reshape(M, M)
    assert rel_fro(T, np.diag(1.0 / np.sqrt(np.diag(Phi).astype(np.float64)))) <= TOL_FP32


def sweeps_of_one_pair(Phi):
    """Sweeps over the up to 32 columns of a pair of blocks until one finds nothing above the tolerance, products carried in
    fp64, with the largest cosine each starts from.  Column i is row i of the Cholesky factor."""
    W = np.zeros((32, Phi.shape[0]))
    W[:len(Phi)] = np.linalg.cholesky(Phi.astype(np.float64)).T
    cosines = []
    while True:
        G, U = W @ W.T, np.eye(32)
        n = np.sqrt(np.maximum(np.diag(G), 1e-300))
        cosines.append(np.abs(G / np.outer(n, n) - np.diag(np.diag(G) / n ** 2)).max())
        if cosines[-1] <= 1e-14:
            return cosines
        for q in range(31):
            R = np.eye(32)
            for k in range(16):
                p, r = 31 if k == 0 else (q + k) % 31, (q - k) % 31
                if G[p, r] ** 2 > 1e-28 * G[p, p] * G[r, r]:
                    d = G[r, r] - G[p, p]
                    t = 0.5 * np.arctan2(np.copysign(2 * G[p, r], G[p, r] if d >= 0 else -G[p, r]), abs(d))
                    R[p, p] = R[r, r] = np.cos(t)
                    R[p, r], R[r, p] = np.sin(t), -np.sin(t)
            G, U = R.T @ G @ R, U @ R
        W = U.T @ W


@pytest.mark.parametrize("decades,seed", [(1, 37), (2, 38), (2, 8), (4, 10)])
def test_products_of_a_visit_are_carried_in_fp64(env, decades, seed):
    """As many sweeps as with all of it in fp64.  The angles are fp32: they leave up to 4 x 2^-24 of a product, which is below the
    tolerance from cosines of 4e-8 on, where these matrices are before their last sweep that rotates.  With products carried in
    fp32 the first two take a sweep more."""
    torch, B = env
    M = 16
    q, _ = np.linalg.qr(np.random.default_rng(1000 * M + seed).standard_normal((M, M)))
    Phi = ((q * np.logspace(0, -decades, M)) @ q.T).astype(np.float32)
    Phi = np.triu(Phi) + np.triu(Phi, 1).T
    cosines = sweeps_of_one_pair(Phi)
    assert cosines[-2] < 4e-8
    L = B.Layer(M, 4, beta=0.0, gamma=1.0)
    L.set(B.FW_F_PHIX, torch.from_numpy(Phi).cuda())
    scratch, nb = scratch_for(torch, B, M)
    B.fw_evd_whiten(L.handle, scratch, nb, 0.0)
    assert L.sync_status() == B.FW_OK
    assert rounds_taken(torch, scratch, M) == len(cosines)
