"""The product out = G B where CTA pairs walk over several tiles: one more tile than a full grid, a last tile of a
few rows, tile counts that leave pairs with unequal shares, widths that are no multiple of the 32-column chunks."""
import numpy as np
import pytest

from oracle import fw_oracle as O

from fwtest_util import TOL_TC, rel_fro, t2n

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
