"""The product out = G B where CTA pairs walk over several tiles: one more tile than a full grid, a last tile of a
few rows, tile counts that leave pairs with unequal shares, widths that are no multiple of the 32-column chunks."""
import numpy as np
import pytest

from oracle import fw_oracle as O

from fwtest_util import TOL_FP32, TOL_TC, rel_fro, t2n

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2010_01546_b200 import binding as B, build
    build.build_library()
    return torch, B


@pytest.mark.parametrize("M,rows", [(16, 256 * 74), (36, 256 * 74 + 1), (64, 256 * 149 + 33), (260, 256 * 75 + 17),
                                    (576, 256 * 50 - 1), (132, 256)])
def test_products_over_many_tiles(env, M, rows):
    torch, B = env
    rng = np.random.default_rng(M + rows)
    L = B.Layer(M, 4, beta=0.0, gamma=1.0, prec=B.FW_PREC_TF32)
    T = (np.eye(M) + 0.5 * rng.standard_normal((M, M)) / np.sqrt(M)).astype(np.float32)
    L.set(B.FW_F_T, torch.from_numpy(T).cuda())
    Lo = O.Layer(M, 4)
    Lo.T = T.astype(np.float64)
    dY = rng.standard_normal((rows, M)).astype(np.float32)
    guard = 64
    buf = torch.full((rows * M + guard,), float("nan"), device="cuda")
    dX = buf[:rows * M].view(rows, M)
    B.fw_whiten_backward(L.handle, torch.from_numpy(dY).cuda(), rows, dX)
    assert rel_fro(t2n(dX), O.whiten_backward(Lo, dY)) <= TOL_TC
    assert bool(torch.isnan(buf[rows * M:]).all())              # nothing past the last row
    assert L.sync_status() == B.FW_OK


@pytest.mark.parametrize("N,M", [(4, 255), (4, 256), (4, 257), (65, 300), (16, 511), (64, 576), (130, 577), (256, 640), (100, 1031), (5, 2050)])
def test_fp32_products_shared_by_a_cluster(env, N, M):
    """Few tiles and a long K: G Qs and the re-sync products on two and four CTAs a tile, uneven shares of K among them, odd
    sizes."""
    torch, B = env
    rng = np.random.default_rng(N + M)
    Phi = rng.standard_normal((M, M)).astype(np.float32)
    Phi = np.triu(Phi) + np.triu(Phi, 1).T
    T = (np.eye(M) + 0.3 * rng.standard_normal((M, M)) / np.sqrt(M)).astype(np.float32)
    G = rng.standard_normal((N, M)).astype(np.float32)
    L = B.Layer(M, N, beta=0.0, gamma=1.0)
    L.set(B.FW_F_PHIX, torch.from_numpy(Phi).cuda())
    L.set(B.FW_F_T, torch.from_numpy(T).cuda())
    B.fw_group_cond_reduce([L.handle], 0, 0)
    T64, P64 = T.astype(np.float64), Phi.astype(np.float64)
    Q = t2n(L.get(B.FW_F_Q)).reshape(M, M)
    Y = t2n(L.get(B.FW_F_PHIY)).reshape(M, M)
    assert rel_fro(Q, T64.T @ T64) <= TOL_FP32 and rel_fro(Y, T64 @ P64 @ T64.T) <= TOL_FP32
    assert np.array_equal(Y, Y.T)
    Gt = t2n(L.grad_transform(torch.from_numpy(G).cuda()))
    assert rel_fro(Gt, G.astype(np.float64) @ Q.astype(np.float64)) <= TOL_FP32
    assert L.sync_status() == B.FW_OK


@pytest.mark.parametrize("dims", [[(27, 67), (603, 67)], [(27, 16)] * 8 + [(603, 16)], [(5, 3), (255, 9), (300, 10), (1, 1)],
                                  [(64, 64), (16, 3), (1031, 5)]])
def test_a_group_whose_longest_k_is_shared(env, dims):
    """Layers of one launch whose K is too short to share beside one whose K is: some CTAs of a short one's clusters have nothing
    to add."""
    torch, B = env
    rng = np.random.default_rng(len(dims) + dims[-1][0])
    Ls, T64, P64, G, W = [], [], [], [], []
    for M, N in dims:
        Phi = rng.standard_normal((M, M)).astype(np.float32)
        Phi = np.triu(Phi) + np.triu(Phi, 1).T
        T = (np.eye(M) + 0.3 * rng.standard_normal((M, M)) / np.sqrt(M)).astype(np.float32)
        L = B.Layer(M, N, beta=0.0, gamma=1.0)
        L.set(B.FW_F_PHIX, torch.from_numpy(Phi).cuda())
        L.set(B.FW_F_T, torch.from_numpy(T).cuda())
        Ls.append(L); T64.append(T.astype(np.float64)); P64.append(Phi.astype(np.float64))
        G.append(torch.from_numpy(rng.standard_normal((N, M)).astype(np.float32)).cuda())
        W.append(torch.zeros((N, M), device="cuda"))
    hs = [L.handle for L in Ls]
    B.fw_group_cond_reduce(hs, 0, 0)
    B.fw_group_grad_transform_step(hs, G, W, None, None, 1.0)
    for i, (L, (M, N)) in enumerate(zip(Ls, dims)):
        Q = t2n(L.get(B.FW_F_Q)).reshape(M, M)
        assert rel_fro(t2n(L.get(B.FW_F_PHIY)).reshape(M, M), T64[i] @ P64[i] @ T64[i].T) <= TOL_FP32
        assert rel_fro(-t2n(W[i]), t2n(G[i]) @ Q) <= TOL_FP32
        assert L.sync_status() == B.FW_OK
