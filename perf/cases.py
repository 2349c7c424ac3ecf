"""The work a user has this library do, as cases that can be timed and compared.

Every case is one training-time pass through the public entry points of
`paper_2010_01546_b200.binding`, on inputs drawn on the GPU from a seed:

  step    one iteration of a set of layers: moments of the batch, K recursion
          steps, gradient transform, parameter step (grouped calls)
  single  the same iteration for one layer through the one-layer calls
  reduce  the recursion alone over independent layers with a given covariance
  evd     whitening from the eigenvalue decomposition (the paper's direct construction)
  whiten  explicit whitening of a batch, forward and backward (the direct method)

A case is a flat dict; `kind` picks one of the above, the other entries are its
sizes and options.  Layer state and parameters live across passes, as in a
training loop.
"""
import math

import torch

from paper_2010_01546_b200 import binding as B
from paper_2010_01546_b200 import synth

DEV = "cuda"
ENGINES = {"fp32": (B.FW_F32, B.FW_PREC_FP32), "tf32": (B.FW_F32, B.FW_PREC_TF32), "bf16": (B.FW_BF16, B.FW_PREC_BF16)}

# The hyper-parameters of the paper's experiments with the recursive method (its Sec. 6; the library's defaults) and
# the ones of the layer-set workloads: no leakage, no smoothing of Q, running covariance with decay 0.9.
PAPER = {"alpha": 0.1, "beta": 0.1, "gamma": 0.99}
PLAIN = {"alpha": 0.9, "beta": 0.0, "gamma": 1.0}


# ----------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------
def cifar_step(batch, engine="tf32", c0=16, depth=5, nhwc=False, momentum=False, K=4, P=16, hyper=PLAIN):
    """3x3 convolutions in three stages of `depth`, c0 / 2 c0 / 4 c0 channels on 32 / 16 / 8 maps (c0 = 16,
    depth = 5: the ResNet-20-shaped set)."""
    return {"kind": "step", "set": "cifar", "batch": batch, "c0": c0, "depth": depth, "engine": engine, "nhwc": nhwc,
            "momentum": momentum, "K": K, "P": P, **hyper}


def imagenet_step(batch, engine="bf16", K=4, P=16):
    """The ResNet-50-shaped set: 1x1 and 3x3 bottleneck convolutions of four stages and the classifier."""
    return {"kind": "step", "set": "imagenet", "batch": batch, "c0": 64, "depth": 1, "engine": engine, "nhwc": False,
            "momentum": False, "K": K, "P": P, **PLAIN}


def ragged_step(batch, width, K=4, P=16):
    """First convolutions and odd-width dense layers: patch lengths that are no multiple of any tile (27 = 3x3x3,
    147 = 7x7x3), odd row counts."""
    return {"kind": "step", "set": "ragged", "batch": batch, "c0": width, "depth": 1, "engine": "tf32", "nhwc": False,
            "momentum": False, "K": K, "P": P, **PLAIN}


def single(M, N, rows, engine, K, P):
    return {"kind": "single", "M": M, "N": N, "rows": rows, "engine": engine, "K": K, "P": P, **PLAIN}


def reduce(M, layers, K, P, cond):
    return {"kind": "reduce", "M": M, "layers": layers, "K": K, "P": P, "cond": cond, **PLAIN}


def evd(c0, depth):
    return {"kind": "evd", "c0": c0, "depth": depth, "g_max": 10.0}


def whiten(M, rows, engine):
    return {"kind": "whiten", "M": M, "rows": rows, "engine": engine}


def listed():
    return [
        # one linear layer of 64 inputs, batch 128: the smallest use, all launches and latency
        dict(single(64, 32, 128, "fp32", 8, 16), name="linear_m64_fp32"),
        # ResNet-20-shaped set on CIFAR-sized maps: the benchmark's default workload, rows already cut
        dict(cifar_step(128), name="resnet20_tf32"),
        # the same set fed with the activations as the network has them
        dict(cifar_step(128, nhwc=True), name="resnet20_nhwc_tf32"),
        # the same set as the paper trains it: leaky transform, smoothed Q, momentum and weight decay
        dict(cifar_step(128, momentum=True, K=1, P=0, hyper=PAPER), name="resnet20_paper_tf32"),
        # the same set on the engine that matches fp64 to 1e-5, smaller batch
        dict(cifar_step(32, engine="fp32"), name="resnet20_fp32"),
        # ResNet-50-shaped set, bf16 activations, batch 256: the largest set
        dict(imagenet_step(256), name="resnet50_bf16"),
        # one wide 3x3 convolution (256 channels on 14x14 maps), batch 256: tensor-bound moments
        dict(single(2304, 256, 256 * 196, "tf32", 8, 16), name="conv_m2304_tf32"),
        # odd sizes: first convolutions and dense layers of odd width
        dict(ragged_step(33, 67), name="ragged_tf32"),
        # recursion over many layers, state on chip (M = 256) and streamed (M = 1152)
        dict(reduce(256, 64, 8, 32, 1e4), name="reduce_m256_x64"),
        dict(reduce(1152, 64, 8, 32, 1e4), name="reduce_m1152_x64"),
        # direct construction of the whitening transform for the ResNet-20-shaped set
        dict(evd(16, 5), name="evd_resnet20"),
        # direct method: every row whitened forward and its gradient sent back
        dict(whiten(576, 32768, "tf32"), name="whiten_m576_tf32"),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    pick = rng.randrange(10)
    if pick == 0:
        M = _log(rng, 16, 400)
        return single(M, _log(rng, 4, 200), _log(rng, 2 * M, 20000), rng.choice(("fp32", "tf32")), rng.randint(1, 8),
                      rng.choice((0, 8, 16)))
    if pick == 1:
        return cifar_step(_log(rng, 8, 160), c0=rng.randint(9, 18), depth=rng.randint(1, 5), K=rng.randint(1, 6),
                          P=rng.choice((4, 8, 16)))
    if pick == 2:
        return cifar_step(_log(rng, 8, 160), c0=4 * rng.randint(2, 5), depth=rng.randint(1, 5), nhwc=True,
                          K=rng.randint(1, 6), P=rng.choice((4, 8, 16)))
    if pick == 3:
        return cifar_step(_log(rng, 16, 160), c0=rng.randint(10, 16), depth=rng.randint(1, 5), momentum=True,
                          K=rng.randint(1, 4), P=rng.choice((0, 0, 4)), hyper=PAPER)
    if pick == 4:
        return cifar_step(_log(rng, 20, 100), engine="fp32", c0=rng.randint(8, 16), depth=rng.randint(1, 5),
                          K=rng.randint(1, 6), P=rng.choice((4, 8, 16)))
    if pick == 5:
        engine = rng.choice(("bf16", "bf16", "tf32"))
        return imagenet_step(_log(rng, 16, 255 if engine == "bf16" else 120), engine=engine, K=rng.randint(1, 4),
                             P=rng.choice((4, 8, 16)))
    if pick == 6:
        M = _log(rng, 640, 3000)
        return single(M, _log(rng, 32, 1000), _log(rng, M, 100000 if M < 2400 else 30000), "tf32", rng.randint(1, 8),
                      rng.choice((4, 8, 16)))
    if pick == 7:
        return ragged_step(2 * _log(rng, 4, 40) + 1, 2 * _log(rng, 12, 60) + 1, K=rng.randint(1, 6),
                           P=rng.choice((4, 8, 16)))
    if pick == 8:
        M = _log(rng, 48, 2304)
        return reduce(M, _log(rng, 1, 64 if M < 1200 else 16), rng.randint(1, 8), rng.choice((0, 8, 16, 32)),
                      10.0 ** rng.randint(2, 5))
    if rng.random() < 0.5:
        return evd(rng.randint(6, 15), rng.randint(1, 4))
    M = _log(rng, 64, 1500)
    return whiten(M, _log(rng, 200, min(100000, 40000000 // M)), rng.choice(("tf32", "tf32", "fp32")))


# ----------------------------------------------------------------------------
# layers of a case
# ----------------------------------------------------------------------------
def _layers(case):
    """(rows, M, N, H, C, k) of every layer of a set."""
    n, c0 = case.get("batch", 1), case["c0"]
    if case["kind"] == "evd" or case["set"] == "cifar":
        return [(n * hw * hw, 9 * c, c, hw, c, 3) for c, hw in ((c0, 32), (2 * c0, 16), (4 * c0, 8))
                for _ in range(case["depth"])]
    if case["set"] == "imagenet":
        return [(*synth.shape_dims(s), s["HW"], s["C_in"], s["k"]) for s in synth.resnet50_shapes(n)]
    return [(n * 31 * 31, 27, c0, 31, 3, 3), (n * 15 * 15, 147, c0, 15, 3, 7), (n * 7 * 7, 9 * c0, c0, 7, c0, 3),
            (n * 63, c0 + 2, 2 * c0 + 1, 1, c0 + 2, 1), (n * 63, 2 * c0 + 1, 10, 1, 2 * c0 + 1, 1)]


def _recursion_flops(M, K, P, stale):
    # per step: column norms, alignment, P iterations, u, t (2 M^2 each), rank-one updates of Q, T and Phi_y
    return K * ((P + 5) * 2.0 * M * M + 8.0 * M * M) + (3.0 * M * M * M if stale else 0.0)


def work(case):
    kind = case["kind"]
    if kind == "evd":
        # read Phi_x, write T, Q, Phi_y, Qs; tridiagonal or Jacobi, about 9 M^3, and three M^3 products
        Ms = [m for _, m, *_ in _layers(case)]
        return {"bytes": sum(24.0 * m * m for m in Ms), "flops": sum(15.0 * m ** 3 for m in Ms)}
    if kind == "whiten":
        M, r = case["M"], case["rows"]
        return {"bytes": 16.0 * r * M + 4.0 * M * M, "flops": 4.0 * r * M * M}
    if kind == "reduce":
        M, n = case["M"], case["layers"]
        # Phi_y, T, Q read and written once
        return {"bytes": n * 24.0 * M * M, "flops": n * _recursion_flops(M, case["K"], case["P"], False)}
    if kind == "single":
        dims = [(case["rows"], case["M"], case["N"], 1, case["M"], 1)]
    else:
        dims = _layers(case)
    size = 2 if case["engine"] == "bf16" else 4
    nbytes = flops = 0.0
    for rows, M, N, H, C, k in dims:
        x = rows * C * 4.0 if case.get("nhwc") else float(rows) * M * size
        # the batch; Phi_x, T, Q (and Qs, T Phi_x where they exist) read and written, Phi_y written; G read, W twice
        state = 28.0 + (8.0 if case["beta"] > 0 else 0.0) + (8.0 if case["gamma"] < 1 else 0.0)
        nbytes += x + state * M * M + 12.0 * N * M + (8.0 * N * M if case.get("momentum") else 0.0)
        flops += float(rows) * M * (M + 1) + _recursion_flops(M, case["K"], case["P"], True) + 2.0 * N * M * M
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "evd":
        return {"rel": 1e-5, "max": 1e-3}          # fp64 decomposition of fp32 data, fp32 results
    if kind == "reduce":
        # fp32; a column whose coherence is within rounding of the threshold may join the start vector or not
        return {"rel": 1e-4, "max": 1e-2}
    if case["engine"] == "fp32":
        return {"rel": 2e-5, "max": 1e-3}
    return {"rel": 5e-3, "max": 0.1}               # TF32 products throughout (bf16 inputs are exact)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _mix(g, C, decades):
    """C x 2C factor of a Wishart channel covariance whose spectrum is widened by `decades`."""
    A = torch.randn((C, 2 * C), generator=g, device=DEV) / math.sqrt(2 * C)
    return A * torch.logspace(0, -decades / 2, C, device=DEV)[:, None]


def _maps(g, n, H, C, decades):
    """n x H x H x C activations: half-normal pixels with correlated channels."""
    A = _mix(g, C, decades)
    out = torch.empty((n, H, H, C), device=DEV)
    step = max(1, (1 << 24) // (H * H * C))
    for i in range(0, n, step):
        m = min(n, i + step) - i
        torch.matmul(torch.randn((m, H, H, 2 * C), generator=g, device=DEV), A.T, out=out[i:i + m])
    return out.abs_()


def _patches(a, k, dtype):
    """Patch rows of the activations, columns ordered (ky, kx, c), zero padding, stride 1."""
    n, H, _, C = a.shape
    a = a.to(dtype)
    if k == 1:
        return a.reshape(n * H * H, C)
    p = torch.nn.functional.pad(a, (0, 0, k // 2, k // 2, k // 2, k // 2))
    x = torch.empty((n, H, H, k, k, C), dtype=dtype, device=DEV)
    for i in range(k):
        for j in range(k):
            x[:, :, :, i, j] = p[:, i:i + H, j:j + H]
    return x.view(n * H * H, k * k * C)


def _basis(g, M, n=1, reflectors=8):
    """Unit vectors of the Householder reflectors of n orthogonal bases."""
    w = torch.randn((reflectors, n, M, 1), generator=g, device=DEV)
    return w / w.norm(dim=2, keepdim=True)


def _gaussian_rows(g, rows, M, cond):
    """Rows ~ N(0, U diag(logspace(0, -log10 cond)) U^T)."""
    x = torch.randn((rows, M), generator=g, device=DEV)
    x *= torch.logspace(0, -math.log10(cond) / 2, M, device=DEV)
    for w in _basis(g, M):
        x -= 2 * (x @ w[0]) @ w[0].T
    return x


def _covariances(g, M, n, cond):
    """n matrices U diag(logspace(0, -log10 cond)) U^T, exactly symmetric, fp32."""
    out = torch.empty((n, M, M), device=DEV)
    out.copy_(torch.diag(torch.logspace(0, -math.log10(cond), M, device=DEV)))
    for w in _basis(g, M, n):
        out -= 2 * w @ (w.mT @ out)
        out -= 2 * (out @ w) @ w.mT
    return torch.triu(out) + torch.triu(out, 1).mT


def _params(g, N, M):
    W = torch.randn((N, M), generator=g, device=DEV) / math.sqrt(M)
    G = torch.randn((N, M), generator=g, device=DEV)
    return W, torch.zeros(N, device=DEV), G, torch.randn(N, generator=g, device=DEV)


def _layer(case, M, N):
    x_dtype, prec = ENGINES[case["engine"]]
    return B.Layer(M, N, device=DEV, x_dtype=x_dtype, prec=prec, alpha=case["alpha"], beta=case["beta"],
                   gamma=case["gamma"])


class State:
    """A user's program between two calls: plain attributes, set by prepare()."""


def prepare(case, seed):
    s = State()
    s.case = case
    g = _gen(seed)
    kind = case["kind"]
    if kind == "step":
        _prepare_step(s, case, g)
    elif kind == "single":
        M, N, rows = case["M"], case["N"], case["rows"]
        s.X = _gaussian_rows(g, rows, M, 1e3 if M < 640 else 1e4)
        s.W, s.b, s.G, s.gb = _params(g, N, M)
        s.layer = _layer(case, M, N)
        s.layer.attach_params(s.W, s.b)
        s.Gt = torch.empty_like(s.G)
    elif kind == "reduce":
        M, n = case["M"], case["layers"]
        phi = _covariances(g, M, n, case["cond"])
        s.layers = [B.Layer(M, 16, device=DEV, alpha=case["alpha"], beta=case["beta"], gamma=case["gamma"])
                    for _ in range(n)]
        for i, L in enumerate(s.layers):
            L.set(B.FW_F_PHIX, phi[i])
        s.handles = [L.handle for L in s.layers]
        s.Q = torch.empty((n, M, M), device=DEV)
    elif kind == "evd":
        s.layers, s.T, s.Q = [], [], []
        for _, M, N, *_ in _layers(case):
            # the EVD method's own settings in the paper's experiments: alpha 0.9, beta 0.95
            L = B.Layer(M, N, device=DEV, prec=B.FW_PREC_TF32, alpha=0.9, beta=0.95, gamma=1.0)
            A = torch.randn((M, 2 * M), generator=g, device=DEV) / math.sqrt(2 * M)
            A *= torch.logspace(0, -1, M, device=DEV)[:, None]
            phi = A @ A.T
            L.set(B.FW_F_PHIX, torch.triu(phi) + torch.triu(phi, 1).T)
            s.layers.append(L)
            s.T.append(torch.empty((M, M), device=DEV))
            s.Q.append(torch.empty((M, M), device=DEV))
        s.handles = [L.handle for L in s.layers]
        s.bytes = [B.fw_evd_scratch_bytes(L.M) for L in s.layers]
        s.scratch = [torch.empty((n + 255) // 256 * 256, dtype=torch.uint8, device=DEV) for n in s.bytes]
    else:
        M, rows = case["M"], case["rows"]
        x_dtype, prec = ENGINES[case["engine"]]
        s.X = _gaussian_rows(g, rows, M, 1e3)
        s.dY = torch.randn((rows, M), generator=g, device=DEV)
        s.Y, s.dX = torch.empty_like(s.X), torch.empty_like(s.X)
        s.layer = B.Layer(M, 16, device=DEV, x_dtype=x_dtype, prec=prec, alpha=0.9, beta=0.0, gamma=1.0)
        T = torch.randn((M, M), generator=g, device=DEV) * (0.5 / math.sqrt(M))
        T.diagonal().add_(1.0)
        s.layer.set(B.FW_F_T, T)
        s.layer.set(B.FW_F_MU, torch.randn(M, generator=g, device=DEV) * 0.1)
    return s


def _prepare_step(s, case, g):
    n = case["batch"]
    dtype = torch.bfloat16 if case["engine"] == "bf16" else torch.float32
    decades = 1.0 if case["set"] == "imagenet" else 0.0
    dims = _layers(case)
    s.X, s.layers, s.W, s.b, s.G, s.gb = [], [], [], [], [], []
    for rows, M, N, H, C, k in dims:
        if H == 1:
            x = _maps(g, rows, 1, C, decades).view(rows, C).to(dtype)
        else:
            a = _maps(g, n, H, C, decades)
            x = a if case["nhwc"] else _patches(a, k, dtype)
        s.X.append(x)
        W, b, G, gb = _params(g, N, M)
        s.W.append(W); s.b.append(b); s.G.append(G); s.gb.append(gb)
        L = _layer(case, M, N)
        L.attach_params(W, b)
        s.layers.append(L)
    s.handles = [L.handle for L in s.layers]
    s.rows = [d[0] for d in dims]
    s.ldx = [d[1] for d in dims]
    if case["nhwc"]:
        s.geometry = [[n] * len(dims)] + [[d[i] for d in dims] for i in (3, 3, 4, 5)]
        s.bytes = [B.fw_nhwc_scratch_bytes(n, H, H, C, k) for _, _, _, H, C, k in dims]
        s.scratch = [torch.empty(b, dtype=torch.uint8, device=DEV) for b in s.bytes]
    if case["momentum"]:
        s.Gt = [torch.empty_like(x) for x in s.G]
        s.vW = [torch.zeros_like(x) for x in s.W]
        s.vb = [torch.zeros_like(x) for x in s.b]


# ----------------------------------------------------------------------------
# one pass
#
# What a step leaves in the caller's hands is the updated W and b (and the
# transformed gradient and velocity where the optimiser is called apart).  They
# depend on all of the layer's state: W on the transform, so on the covariance,
# the powers and every recursion step, b on the running mean.
# ----------------------------------------------------------------------------
def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "step":
        if case["nhwc"]:
            B.fw_group_cov_update_nhwc(s.handles, s.X, *s.geometry, s.scratch, s.bytes)
        else:
            B.fw_group_cov_update(s.handles, s.X, s.rows, s.ldx)
        B.fw_group_cond_reduce(s.handles, case["K"], case["P"])
        if case["momentum"]:
            for L, W, b, G, gb, Gt, vW, vb in zip(s.layers, s.W, s.b, s.G, s.gb, s.Gt, s.vW, s.vb):
                L.grad_transform(G, Gt)
                B.fw_step_momentum(L.handle, W, b, Gt, gb, vW, vb, 0.1, 0.9, 5e-4)
            return {"W": s.W, "b": s.b, "Gt": s.Gt, "vW": s.vW}
        B.fw_group_grad_transform_step(s.handles, s.G, s.W, s.b, s.gb, 0.1)
        return {"W": s.W, "b": s.b}
    if kind == "single":
        L = s.layer
        L.cov_update(s.X)
        L.cond_reduce(case["K"], case["P"])
        L.grad_transform(s.G, s.Gt)
        L.step(s.W, s.b, s.Gt, s.gb, 0.1)
        return {"W": s.W, "b": s.b, "Gt": s.Gt}
    if kind == "reduce":
        B.fw_group_cond_reduce(s.handles, case["K"], case["P"])
        size = case["M"] * case["M"] * 4
        for i, h in enumerate(s.handles):
            B.fw_layer_get(h, B.FW_F_QS, s.Q[i], size)
        return s.Q
    if kind == "evd":
        B.fw_group_evd_whiten(s.handles, s.scratch, s.bytes, case["g_max"])
        for L, T, Q in zip(s.layers, s.T, s.Q):
            B.fw_layer_get(L.handle, B.FW_F_T, T, T.numel() * 4)
            B.fw_layer_get(L.handle, B.FW_F_QS, Q, Q.numel() * 4)
        return {"T": s.T, "Qs": s.Q}
    B.fw_whiten_forward(s.layer.handle, s.X, case["rows"], s.Y)
    B.fw_whiten_backward(s.layer.handle, s.dY, case["rows"], s.dX)
    return {"Y": s.Y, "dX": s.dX}
