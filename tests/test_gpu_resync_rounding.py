"""Re-sync products Phi_y = T Phi_x T^T of the tensor-core engine against the same products in 64 bits with every operand and the
intermediate product rounded to TF32, nearest, at the place where the engine rounds: one layer and groups of mixed sizes that take more than
one launch."""
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


def tf32(A):
    """Nearest, ties away from zero, of numbers far from overflow."""
    bits = np.ascontiguousarray(A, np.float32).view(np.uint32)
    return ((bits + np.uint32(0x1000)) & np.uint32(0xffffe000)).view(np.float32).astype(np.float64)


def tolerance(M):
    """Relative, in the Frobenius norm.  A chain of M / 8 accumulations loses at most a = (M / 8) 2^-23 of a well-conditioned product.  Where
    a moves an entry of the first product over the middle of two TF32 numbers, the entry is off by a step, 2^-10 of it: a share
    2 a / 2^-10 of the entries, or a few of them.  (Operands that are cut off instead of rounded: 4.8e-4 and more.)"""
    a = M / 8 * 2.0 ** -23
    return 2 * a + np.sqrt(max(2 * a * 2.0 ** 10, 4 / M ** 2)) * 2.0 ** -10


@pytest.mark.parametrize("gamma", [1.0, 0.99])
@pytest.mark.parametrize("sizes", [[16], [100], [128], [600], [1020], [1028], [1100],
                                   [20, 36, 48, 64, 100, 128, 132, 144, 160, 200, 256, 260, 288, 300, 576, 16, 24, 32, 96, 400],
                                   [1040, 144, 1100, 288, 1344]])
def test_products_are_rounded_to_nearest(env, sizes, gamma):
    torch, B = env
    rng = np.random.default_rng(sum(sizes))
    cu = lambda a: torch.from_numpy(a).cuda()
    data = []
    for M in sizes:
        A = rng.standard_normal((M, M + 8)) / np.sqrt(M)
        P = (A @ A.T).astype(np.float32)
        T = (np.eye(M) + 0.3 * rng.standard_normal((M, M)) / np.sqrt(M)).astype(np.float32)
        L = B.Layer(M, 4, beta=0.0, gamma=gamma, prec=B.FW_PREC_TF32)
        L.set(B.FW_F_T, cu(T))
        L.set(B.FW_F_PHIX, cu(np.triu(P) + np.triu(P, 1).T))
        data.append((M, L, T, np.triu(P) + np.triu(P, 1).T))
    B.fw_group_cond_reduce([L.handle for _, L, _, _ in data], 0, 0)
    for M, L, T, P in data:
        Tr = tf32(T)
        want = np.triu(Tr @ tf32(tf32(P) @ Tr.T))
        want += np.triu(want, 1).T                     # the lower triangle is the upper one's image
        got = t2n(L.get(B.FW_F_PHIY)).reshape(M, M).astype(np.float64)
        assert np.linalg.norm(got - want) <= tolerance(M) * np.linalg.norm(want)
        assert np.array_equal(got, got.T)
        assert L.sync_status() == B.FW_OK
