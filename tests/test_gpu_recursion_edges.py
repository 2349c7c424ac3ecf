"""On-chip recursion at the edges of its register tiles (rows of 128 entries per trip, one or two groups of four rows
per warp, one or several CTAs per layer) and of its step batches (T and Q take eight steps at a time)."""
import numpy as np
import pytest

from oracle import fw_oracle as O
from paper_2010_01546_b200 import synth

from test_gpu_recursion_rounding import Reference
from fwtest_util import TOL_FP32, group_reduce_with_replay, oracle_hyper, reduce_with_replay, rel_fro, t2n

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2010_01546_b200 import binding as B, build
    build.build_library()
    return torch, B


def spd32(M, cond, seed):
    Phi, _, _ = synth.spd_with_spectrum(M, cond, seed, basis="qr" if M <= 300 else "householder")
    P = Phi.astype(np.float32)
    return np.triu(P) + np.triu(P, 1).T


def check(L, Lo, B):
    for f, ref in ((B.FW_F_T, Lo.T), (B.FW_F_Q, Lo.Q), (B.FW_F_QS, Lo.Qs), (B.FW_F_PHIY, Lo.phiy())):
        assert rel_fro(t2n(L.get(f)).reshape(ref.shape), ref) <= TOL_FP32


@pytest.mark.parametrize("M", [1, 4, 63, 64, 65, 128, 129, 255, 256, 257, 384, 513, 624])
def test_tile_edges(env, M):
    torch, B = env
    Phi = spd32(M, 1e2, 900 + M)
    La, Lb = B.Layer(M, 4, beta=0.2, gamma=1.0), B.Layer(M, 4, beta=0.2, gamma=1.0)
    Lo = O.Layer(M, 4, oracle_hyper(La.desc))
    for L in (La, Lb):
        L.set(B.FW_F_PHIX, torch.from_numpy(Phi).cuda())
    Lo.set_phix(Phi)
    reduce_with_replay(La, Lo, 2, 3, B, torch)
    check(La, Lo, B)
    # 18 steps of one call (batches of 8, 8 and 2) are those of single calls, Q_s apart (smoothed once per call)
    for _ in range(16):
        La.cond_reduce(1, 3)
    Lb.cond_reduce(18, 3)
    for f in (B.FW_F_T, B.FW_F_Q, B.FW_F_PHIY, B.FW_F_ALIGN_W):
        assert torch.equal(La.get(f), Lb.get(f))
    assert La.sync_status() in (B.FW_OK, B.FW_WARN_NO_SUBSPACE)


@pytest.mark.parametrize("dims", [[256] * 64, [620, 577, 300, 145, 64, 33, 1], [128, 12]])
def test_groups(env, dims):
    torch, B = env
    Ls, Los = [], []
    for i, M in enumerate(dims):
        Phi = spd32(M, 1e2, 40 + i)
        L = B.Layer(M, 4, beta=0.0, gamma=1.0)
        Lo = O.Layer(M, 4, oracle_hyper(L.desc))
        L.set(B.FW_F_PHIX, torch.from_numpy(Phi).cuda()); Lo.set_phix(Phi)
        Ls.append(L); Los.append(Lo)
    if len(dims) > 8:                       # a full group: every layer must come out as it does alone
        B.fw_group_cond_reduce([L.handle for L in Ls], 2, 4)
        for i in (0, 27, 28, 63):
            L = B.Layer(dims[i], 4, beta=0.0, gamma=1.0)
            L.set(B.FW_F_PHIX, torch.from_numpy(spd32(dims[i], 1e2, 40 + i)).cuda())
            reduce_with_replay(L, Los[i], 2, 4, B, torch)
            check(Ls[i], Los[i], B)
            assert torch.equal(Ls[i].get(B.FW_F_T), L.get(B.FW_F_T))
        return
    group_reduce_with_replay(Ls, Los, 2, 4, B, torch)
    for L, Lo in zip(Ls, Los):
        check(L, Lo, B)


# ---- layers past the on-chip kernel: teams of CTAs, rows in shared memory or (4001) partly streamed ----
@pytest.mark.parametrize("M,K", [(625, 18), (626, 2), (900, 2), (1153, 2), (1284, 2), (4001, 1)])
def test_team_edges(env, M, K):
    torch, B = env
    Phi = spd32(M, 1e2, 900 + M)
    La, Lb = B.Layer(M, 4, beta=0.2, gamma=1.0), B.Layer(M, 4, beta=0.2, gamma=1.0)
    Lo = O.Layer(M, 4, oracle_hyper(La.desc))
    for L in (La, Lb):
        L.set(B.FW_F_PHIX, torch.from_numpy(Phi).cuda())
    Lo.set_phix(Phi)
    reduce_with_replay(La, Lo, min(K, 2), 3, B, torch)
    check(La, Lo, B)
    for _ in range(K - 2):
        La.cond_reduce(1, 3)
    Lb.cond_reduce(K, 3)                     # 18 steps: T and Q take them in batches of 16 and 2
    for f in (B.FW_F_T, B.FW_F_Q, B.FW_F_PHIY, B.FW_F_ALIGN_W):
        assert torch.equal(La.get(f), Lb.get(f))
    assert La.sync_status() == B.FW_OK


def test_team_waves(env):
    torch, B = env
    dims = [1152] * 7 + [700, 640, 2048, 2048, 100]      # more rows than the chip holds at once, and an on-chip layer
    Ls = []
    for i, M in enumerate(dims):
        L = B.Layer(M, 4, beta=0.0, gamma=1.0)
        L.set(B.FW_F_PHIX, torch.from_numpy(spd32(M, 1e2, 40 + i)).cuda())
        Ls.append(L)
    for _ in range(2):
        B.fw_group_cond_reduce([L.handle for L in Ls], 2, 4)
    for i in (0, 6, 7, 8, 10, 11):
        Phi = torch.from_numpy(spd32(dims[i], 1e2, 40 + i)).cuda()
        L = B.Layer(dims[i], 4, beta=0.0, gamma=1.0)
        L.set(B.FW_F_PHIX, Phi)
        L.cond_reduce(2, 4)
        L.cond_reduce(2, 4)
        for f in (B.FW_F_T, B.FW_F_Q, B.FW_F_PHIY):       # whatever the team
            assert torch.equal(Ls[i].get(f), L.get(f))
        assert Ls[i].sync_status() == B.FW_OK
        if i in (6, 8, 10):                               # and against the operations spelled out (M > 624)
            R = Reference(torch, Phi, L.get(B.FW_F_LAMBDA_BAR)[0], L.desc)
            for _ in range(4):
                R.step(4)
            assert torch.equal(Ls[i].get(B.FW_F_T), R.T.T)


@pytest.mark.parametrize("M,K", [(700, 3), (1153, 18), (256, 3)])
def test_replayed_calls(env, M, K):
    """A pass replayed from a captured graph goes on from the state the pass before left, as a call does: the packet
    exchanges of a team carry numbers that must not come again."""
    torch, B = env
    X = torch.randn(4, 2 * M, M, device="cuda") * torch.logspace(0, -1, M, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    La, Lb = (B.Layer(M, 4, alpha=0.5, beta=0.2, gamma=1.0, stream=stream.cuda_stream) for _ in range(2))
    x = X[0].clone()
    graph = torch.cuda.CUDAGraph()

    def run(L, i):
        with torch.cuda.stream(stream):
            x.copy_(X[i])
            L.cov_update(x)
            L.cond_reduce(K, 2)

    for i in range(4):
        run(La, i)
    for i in range(2):
        run(Lb, i)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        Lb.cov_update(x)
        Lb.cond_reduce(K, 2)
    for i in range(2, 4):
        with torch.cuda.stream(stream):
            x.copy_(X[i])
            graph.replay()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for f in (B.FW_F_PHIX, B.FW_F_T, B.FW_F_Q, B.FW_F_QS, B.FW_F_PHIY, B.FW_F_ALIGN_W):
            assert torch.equal(La.get(f), Lb.get(f))
    assert La.sync_status() == Lb.sync_status() == B.FW_OK
