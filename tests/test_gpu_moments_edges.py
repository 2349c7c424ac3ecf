"""Moment kernels at the edges of their 32 x 32 tiles and of the four entries a thread takes: sizes that are whole float4s and
sizes that are not, few and many row splits, first and later blocks, blocks over two calls."""
import numpy as np
import pytest

from oracle import fw_oracle as O

from fwtest_util import TOL_FP32, TOL_TC, oracle_hyper, rel_fro, t2n

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2010_01546_b200 import binding as B, build
    build.build_library()
    return torch, B


@pytest.mark.parametrize("engine", ["fp32", "tf32"])
@pytest.mark.parametrize("M,rows", [(1, 40), (3, 65), (4, 5000), (31, 900), (32, 20000), (33, 901), (36, 4097), (66, 12000), (129, 700),
                                    (132, 9000), (577, 1200), (1028, 600), (1030, 1100)])
def test_moments_over_two_blocks(env, M, rows, engine):
    torch, B = env
    rng = np.random.default_rng(M + rows)
    L = B.Layer(M, 4, alpha=0.7, beta=0.0, gamma=1.0, prec=B.FW_PREC_FP32 if engine == "fp32" else B.FW_PREC_TF32)
    Lo = O.Layer(M, 4, oracle_hyper(L.desc))
    tol = TOL_FP32 if engine == "fp32" else TOL_TC
    A = rng.standard_normal((M, M)) / np.sqrt(M)
    for block in range(2):
        X = np.abs(rng.standard_normal((rows, M)) @ A).astype(np.float32)
        if block:
            h = rows // 3
            B.fw_cov_update(L.handle, torch.from_numpy(X[:h]).cuda(), h, M, B.FW_COV_ACCUMULATE)
            B.fw_cov_update(L.handle, torch.from_numpy(X[h:]).cuda(), rows - h, M, B.FW_COV_COMMIT)
        else:
            L.cov_update(torch.from_numpy(X).cuda())
        O.cov_update(Lo, X)
        P = t2n(L.get(B.FW_F_PHIX)).reshape(M, M)
        assert np.array_equal(P, P.T)
        assert rel_fro(P, Lo.Phix) <= tol
        assert rel_fro(t2n(L.get(B.FW_F_MU)), Lo.mu) <= tol and rel_fro(t2n(L.get(B.FW_F_PHI_DIAG)), Lo.phi) <= tol
        assert abs(float(L.get(B.FW_F_LAMBDA_BAR)[0]) - Lo.lam_bar) <= tol * abs(Lo.lam_bar)
    assert L.sync_status() == B.FW_OK
