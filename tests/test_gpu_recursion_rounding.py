"""Rounding of the recursion of large layers (M > 624).  A column within rounding of the coherence threshold joins the start
vector or not, so results hold only while every operation is rounded in one way: the kernels are compared bit for bit with
the same operations spelled out in torch (fp64 products in the order of the rows' sums, fp32 elsewhere), and at condition
1e4 their decisions with the oracle's on the device's own Phi_y."""
import numpy as np
import pytest

from oracle import fw_oracle as O
from paper_2010_01546_b200 import synth

from fwtest_util import t2n

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2010_01546_b200 import binding as B, build
    build.build_library()
    return torch, B


def spd32(M, cond, seed):
    Phi, _, _ = synth.spd_with_spectrum(M, cond, seed, basis="householder")
    P = Phi.astype(np.float32)
    return np.triu(P) + np.triu(P, 1).T


class Reference:
    """The operations of a call, one rounding each.  fma(a, b, c) of fp32 numbers is formed in fp64 (the product is exact)
    and rounded to fp32."""

    def __init__(self, torch, Phi, lam_bar, desc):
        self.torch, self.Y, self.lam_bar, self.d = torch, Phi.clone(), lam_bar, desc
        self.M = M = Phi.shape[0]
        self.T = torch.eye(M, device="cuda")            # T^T
        self.Q = torch.eye(M, device="cuda")
        self.width = 4 if M % 4 == 0 else 1             # entries a lane takes at a time

    def fma(self, a, b, c):
        return (a.double() * b.double() + c.double()).float()

    def rows(self, A, x):
        """A x: lanes take the entries of every 32nd float4 (or entry) in ascending order; butterfly from 16 to 1."""
        torch, w = self.torch, self.width
        n = 32 * w
        pad = (-self.M) % n
        A = torch.nn.functional.pad(A, (0, pad)).double().view(A.shape[0], -1, 32, w)
        x = x if x.dim() == 2 else x.expand(A.shape[0], -1)
        x = torch.nn.functional.pad(x, (0, pad)).double().view(A.shape[0], -1, 32, w)
        acc = torch.zeros(A.shape[0], 32, dtype=torch.float64, device="cuda")
        for t in range(A.shape[1]):
            for e in range(w):
                acc = acc + A[:, t, :, e] * x[:, t, :, e]
        lane = torch.arange(32, device="cuda")
        for o in (16, 8, 4, 2, 1):
            acc = acc + acc[:, lane ^ o]
        return acc[:, 0].float()

    def total(self, a, b):
        """a.b in fp32: entry m to thread m mod 1024, butterflies of 32 threads, their sums in ascending order; where M is
        no multiple of four, pairs of entries, eight pairs in order, partial sum p to thread p mod 256, and so on."""
        torch, M = self.torch, self.M
        lane = torch.arange(32, device="cuda")

        def warps(s):
            s = s.view(-1, 32)
            for o in (16, 8, 4, 2, 1):
                s = s + s[:, lane ^ o]
            t = torch.zeros((), device="cuda")
            for v in s[:, 0]:
                t = t + v
            return t

        if self.width == 4:
            pad = (-M) % 1024
            a, b = (torch.nn.functional.pad(v, (0, pad)).view(-1, 1024) for v in (a, b))
            s = torch.zeros(1024, device="cuda")
            for i in range(a.shape[0]):
                s = self.fma(a[i], b[i], s)
            return warps(s)
        pad = (-M) % 4096
        a, b = (torch.nn.functional.pad(v, (0, pad)).view(-1, 8, 2) for v in (a, b))
        q = self.fma(a[..., 1], b[..., 1], a[..., 0] * b[..., 0])
        p = torch.zeros(q.shape[0], device="cuda")
        for i in range(8):
            p = p + q[:, i]
        s = torch.zeros(256, device="cuda")
        for part in p.view(-1, 256):
            s = s + part
        return warps(s)

    def inv_norm(self, n2):
        r = self.torch.rsqrt(n2)
        return r * self.fma(-(0.5 * n2 * r), r, self.torch.full_like(r, 1.5))

    def step(self, P):
        torch, d, Y = self.torch, self.d, self.Y
        f32 = lambda v: torch.tensor(v, dtype=torch.float32, device="cuda")
        xi2 = self.rows(Y, Y)
        mp = int(torch.argmax(xi2))
        c = self.rows(Y, Y[mp])
        thr = torch.maximum(f32(d.c_rel) * xi2[mp].sqrt() * xi2.sqrt(), f32(d.c_abs))
        keep = c.abs() >= thr
        cnt = int(keep.sum())
        w = torch.where(keep, 1.0 / c, torch.zeros_like(c))
        x = self.rows(Y, w) * (f32(1.0) / f32(float(cnt)))
        for _ in range(P):
            x = self.rows(Y, x * self.inv_norm(self.total(x, x)))
        v = x * self.inv_norm(self.total(x, x))
        u = self.rows(Y, v)
        lam = self.total(v, u)
        g = f32(d.delta) * self.lam_bar / torch.maximum(lam, f32(d.eps))
        a = g.sqrt() - 1.0
        a2l = a * a * lam
        vi, vj, ui, uj = v[:, None], v[None, :], u[:, None], u[None, :]
        self.Y = Y + (a * (vi * uj + ui * vj) + a2l * (vi * vj))
        t = self.rows(self.T, v)
        self.T = self.fma((a * t)[:, None], vj, self.T)
        self.Q = self.Q + a * (a + 2.0) * (t[:, None] * t[None, :])
        return torch.stack([lam, g, f32(float(cnt)), f32(float(mp))])


@pytest.mark.parametrize("M,K,P", [(625, 2, 3), (628, 3, 4), (640, 2, 17), (1152, 3, 4), (1153, 2, 5), (2304, 2, 4), (4608, 1, 2)])
def test_bits(env, M, K, P):
    torch, B = env
    Phi = torch.from_numpy(spd32(M, 1e4, 7 + M)).cuda()
    L = B.Layer(M, 4, beta=0.0, gamma=1.0)
    L.set(B.FW_F_PHIX, Phi)
    R = Reference(torch, Phi, L.get(B.FW_F_LAMBDA_BAR)[0], L.desc)
    trace = torch.zeros(K, 4, device="cuda")
    L.cond_reduce(K, P, trace)
    want = torch.stack([R.step(P) for _ in range(K)])
    assert torch.equal(trace, want)
    for f, ref in ((B.FW_F_PHIY, R.Y), (B.FW_F_T, R.T.T), (B.FW_F_Q, R.Q)):
        assert torch.equal(L.get(f).view(M, M), ref)
    assert L.sync_status() == B.FW_OK


@pytest.mark.parametrize("M", [640, 1284, 1301, 3076])
def test_rows_of_t_in_the_order_of_record(env, M):
    """Rows of T^T whose squares overflow fp32 (no bound on their sums' difference between orders) or that come near its
    largest number take their sums in the order of record, as rows whose rounding is open do."""
    torch, B = env
    Phi = torch.from_numpy(spd32(M, 1e2, M)).cuda()
    g = torch.Generator(device="cuda")
    g.manual_seed(M)
    T = torch.eye(M, device="cuda")
    T[:, 3:6] = torch.randn((M, 3), generator=g, device="cuda") * 1e36
    L = B.Layer(M, 4, beta=0.0, gamma=1.0)
    L.set(B.FW_F_PHIX, Phi)
    L.set(B.FW_F_T, T)
    L.set(B.FW_F_PHIY, Phi)
    R = Reference(torch, Phi, L.get(B.FW_F_LAMBDA_BAR)[0], L.desc)
    R.T = T.T.contiguous()
    L.cond_reduce(2, 2)
    for _ in range(2):
        R.step(2)
    got = L.get(B.FW_F_T).view(M, M)
    assert bool(torch.isfinite(got).all()) and torch.equal(got, R.T.T)


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_nonfinite_state(env, bad):
    """A row with an infinity or a NaN reaches every result, as fp32 arithmetic has it, and is reported."""
    torch, B = env
    M = 700
    Phi = torch.from_numpy(spd32(M, 1e2, 3)).cuda()
    Phi[5, 9] = Phi[9, 5] = bad
    L = B.Layer(M, 4, beta=0.0, gamma=1.0)
    L.set(B.FW_F_PHIX, Phi)
    trace = torch.zeros(1, 4, device="cuda")
    L.cond_reduce(1, 2, trace)
    assert not bool(torch.isfinite(trace[0, 0]))
    assert torch.equal(L.get(B.FW_F_PHIY).view(M, M).nan_to_num(1e30, 2e30), Phi.nan_to_num(1e30, 2e30))    # no step taken
    assert L.sync_status() == B.FW_WARN_NONFINITE


@pytest.mark.parametrize("M,seed", [(1152, 1), (1152, 2), (900, 3)])
def test_decisions_at_condition_1e4(env, M, seed):
    torch, B = env
    L = B.Layer(M, 4, beta=0.0, gamma=1.0)
    L.set(B.FW_F_PHIX, torch.from_numpy(spd32(M, 1e4, seed)).cuda())
    trace = torch.zeros(1, 4, device="cuda")
    for _ in range(6):
        L.cond_reduce(0, 0)                       # Phi_y of the first step
        Y = t2n(L.get(B.FW_F_PHIY)).reshape(M, M)
        est = O.principal_subspace(Y, L.desc.c_rel, L.desc.c_abs, O.INIT_ALIGN)
        v = est["v"]
        for _ in range(4):
            v = Y @ v
            v /= np.linalg.norm(v)
        L.cond_reduce(1, 4, trace)
        lam, _, cnt, mp = t2n(trace)[0]
        assert int(mp) == est["m_prime"] and int(cnt) == int(est["mask"].sum())
        # vectors are fp32: lambda_e = v.Y v is off by 2^-24 of ||Y|| per rounded entry, far below sqrt(M) of them together
        assert abs(lam - v @ Y @ v) <= np.sqrt(M) * 2.0 ** -24 * np.linalg.norm(Y, 2)
