"""NaNs that the GPU's own arithmetic makes (all mantissa bits set) through the roundings to TF32: the centred Gram pass of
short blocks, the stored copy of T, both operands and the result of the re-sync products."""
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


def hits(A, c):
    """Row and column c of A are not finite, the rest is."""
    bad = ~np.isfinite(A)
    want = np.zeros_like(bad)
    want[c, :] = want[:, c] = True
    return np.array_equal(bad, want)


@pytest.mark.parametrize("M,rows,at", [(64, 900, 3), (96, 900, 700), (288, 1500, 1400), (576, 700, 650), (1040, 600, 590)])
def test_nan_in_a_short_block(env, M, rows, at):
    torch, B = env
    rng = np.random.default_rng(M)
    X = rng.standard_normal((rows, M)).astype(np.float32)
    X[at, 17] = np.nan                        # below or past the rows that the pilot mean samples
    L = B.Layer(M, 4, alpha=0.5, beta=0.0, gamma=1.0, prec=B.FW_PREC_TF32)
    L.cov_update(torch.from_numpy(X).cuda())
    assert L.sync_status() == B.FW_WARN_NONFINITE
    assert hits(t2n(L.get(B.FW_F_PHIX)).reshape(M, M), 17)
    assert np.array_equal(np.isnan(t2n(L.get(B.FW_F_MU))), np.arange(M) == 17)


@pytest.mark.parametrize("bits", [0x7fffffff, 0xffffffff, 0x7f800001, 0x7f801fff, 0x7fc00000, 0x7f800000])
@pytest.mark.parametrize("gamma", [1.0, 0.99])
@pytest.mark.parametrize("M", [96, 1040])
def test_nan_through_the_resync_products(env, M, gamma, bits):
    torch, B = env
    rng = np.random.default_rng(M)
    bad = np.array([bits], np.uint32).view(np.float32)[0]
    T = (np.eye(M) + 0.3 * rng.standard_normal((M, M)) / np.sqrt(M)).astype(np.float32)
    cu = lambda a: torch.from_numpy(a).cuda()

    def fresh(T, Phi):
        L = B.Layer(M, 4, beta=0.0, gamma=gamma, prec=B.FW_PREC_TF32)
        L.set(B.FW_F_T, cu(T))
        L.set(B.FW_F_PHIX, cu(Phi))
        return L

    # in Phi_x: every entry of T Phi_x T^T depends on it
    Phi = np.eye(M, dtype=np.float32)
    Phi[5, 5] = bad
    L = fresh(T, Phi)
    assert not np.isfinite(t2n(L.get(B.FW_F_PHIY))).any()
    L.cond_reduce(1, 2)
    assert L.sync_status() == B.FW_WARN_NONFINITE
    # in T: a row and a column of Phi_y
    Tb = T.copy()
    Tb[7, 9] = bad
    L = fresh(Tb, np.eye(M, dtype=np.float32))
    assert hits(t2n(L.get(B.FW_F_PHIY)).reshape(M, M), 7)
