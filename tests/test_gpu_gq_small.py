"""The gradient transform of small tensor-core layers: rows and columns past a tile, K shares of one to eight CTAs that end
unevenly, the sizes on both sides of the rule that picks the kernel; products, steps, and what is not finite."""
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


def layer(torch, B, rng, N, M):
    L = B.Layer(M, N, beta=0.0, gamma=1.0, prec=B.FW_PREC_TF32)
    T = (np.eye(M) + 0.3 * rng.standard_normal((M, M)) / np.sqrt(M)).astype(np.float32)
    L.set(B.FW_F_T, torch.from_numpy(T).cuda())
    return L, t2n(L.get(B.FW_F_QS)).reshape(M, M).astype(np.float64)


@pytest.mark.parametrize("N,M", [(1, 16), (16, 20), (17, 168), (32, 172), (33, 336), (64, 340), (65, 100), (64, 576), (128, 576),
                                 (72, 648), (100, 672), (20, 676), (31, 1000), (64, 1024), (128, 1024), (129, 64), (8, 1028)])
def test_small_products_and_steps(env, N, M):
    """Both operands lose up to 2^-10 of a value to TF32 and a chain of M additions at most 2^-22 an addition."""
    torch, B = env
    rng = np.random.default_rng(1000 * N + M)
    L, Q = layer(torch, B, rng, N, M)
    cu = lambda a: torch.from_numpy(a).cuda()
    G, W = (rng.standard_normal((N, M)).astype(np.float32) for _ in range(2))
    b = gb = np.zeros(N, np.float32)
    ref, scale = G.astype(np.float64) @ Q, np.abs(G).astype(np.float64) @ np.abs(Q)
    tol = (2.05 * 2.0 ** -10 + M * 2.0 ** -22) * scale
    guard = torch.full((N * M + 64,), float("nan"), device="cuda")
    out = guard[:N * M].view(N, M)
    L.grad_transform(cu(G), out)
    assert np.all(np.abs(t2n(out) - ref) <= tol)
    assert bool(torch.isnan(guard[N * M:]).all())
    Wd = cu(W)
    B.fw_group_grad_transform_step([L.handle], [cu(G)], [Wd], [cu(b)], [cu(gb)], 0.5)
    assert np.all(np.abs(t2n(Wd) - (W - 0.5 * ref)) <= 0.5 * tol + 2.0 ** -23 * np.abs(W))
    assert L.sync_status() == B.FW_OK
    G[N - 1, M - 1] = np.nan
    L.grad_transform(cu(G), out)
    y = t2n(out)
    assert np.isnan(y[N - 1]).all() and np.isfinite(y[:N - 1]).all()
    assert L.sync_status() == B.FW_WARN_NONFINITE
