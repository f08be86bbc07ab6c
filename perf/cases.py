"""Workloads of this library, each through its public entry points.

Four are whole calls (single pairs, a parameter sweep, the symmetric form),
the rest are the blocks that a program of its own is built from: losses with
their gradients, the adjoints, the field smoother, the optimiser step and one
iteration of a hand-written loop.  Inputs follow the recipes of
paper_2404_01249_gb300/synth.py, drawn on the GPU: brain-like Voronoi pairs,
cell-like spots, Gaussian blobs.

exact() evaluates the same formulas in 64 bits with plain torch.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2404_01249_gb300 import fa

BRAIN = dict(scales="4,2,1", iters="200,100,50")     # the brain pair's schedule
BLOBS = dict(scales="2,1", iters="50,25")            # the small pair's schedule
CELLS = dict(scales="8,4,2,1", iters="200,200,100,50")  # the microscopy schedule
HALF_BRAIN = dict(scales="2,1", iters="100,50")      # its two finer levels on a smaller grid
SVF_STEPS = 7


def listed():
    return [
        # the smallest whole call: 32^3, 75 iterations, all launches and latency
        dict(name="pair_blobs_32", op="pair", image="blobs", D=32, H=32, W=32, window=5,
             storage="f32", state="f32", field="f32", **BLOBS),
        # the headline workload: one brain-MRI-shaped pair, three levels, FP32
        dict(name="pair_brain_160x192x224", op="pair", image="voronoi", D=160, H=192, W=224,
             window=5, storage="f32", state="f32", field="f32", **BRAIN),
        # microscopy: window 7, four levels, 16-bit images, moments and displacement
        dict(name="pair_cells_128x256x256", op="pair", image="cells", D=128, H=256, W=256,
             window=7, storage="bf16", state="bf16", field="f16", **CELLS),
        # a hyper-parameter sweep: uneven brain-like pairs x three learning rates, BF16
        dict(name="sweep_3x3_uneven", op="sweep", image="voronoi", D=131, H=157, W=143, pairs=3,
             settings=3, window=5, storage="bf16", state="bf16", field="f32", **BRAIN),
        # symmetric registration of a pair at the small end of the uneven brain grids
        dict(name="symmetric_96x113x101", op="symmetric", image="voronoi", D=96, H=113, W=101,
             window=5, **HALF_BRAIN),
        # one step of an optimiser in the Lie algebra: loss, gradient and exp(v)
        dict(name="svf_grad_160x192x224", op="svf", image="voronoi", D=160, H=192, W=224,
             window=5, steps=SVF_STEPS),
        # template building: the loss and its gradients for the field and the template
        dict(name="adjoint_160x192x224", op="adjoint", image="voronoi", D=160, H=192, W=224,
             window=5, fixed_grad=False),
        # the LNCC loss as a layer with both gradients, on an uneven grid
        dict(name="lncc_127x181x159", op="lncc", image="voronoi", D=127, H=181, W=159, window=5,
             both=True),
        # the mutual-information loss as a layer
        dict(name="mi_160x192x224", op="mi", image="voronoi", D=160, H=192, W=224, bins=32),
        # the regulariser of a displacement field
        dict(name="smooth_160x192x224", op="smooth", D=160, H=192, W=224, channels=3, sigma=1.0),
        # the optimiser's step on a whole field
        dict(name="step_160x192x224", op="step", D=160, H=192, W=224, moments="f32"),
        # one iteration of a loop written from the per-step calls, on a small odd grid
        dict(name="loop_37x45x53", op="loop", image="voronoi", D=37, H=45, W=53, window=5,
             sigma_grad=1.0, sigma_warp=0.5),
    ]


def _grid(rng, lo, hi):
    """A grid of about lo..hi voxels (log-uniform), any size on each axis."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    a = [math.exp(rng.uniform(-0.35, 0.35)) for _ in range(3)]
    g = (n / (a[0] * a[1] * a[2])) ** (1.0 / 3.0)
    D, H, W = (max(8, int(round(g * k))) for k in a)
    while D * H * W > hi:
        D, H, W = max(8, D - 1), max(8, H - 1), max(8, W - 1)
    return dict(D=D, H=H, W=W)


def draw(rng):
    op = rng.choice(("pair", "pair", "cells", "sweep", "symmetric", "svf", "adjoint", "lncc", "mi",
                     "smooth", "step", "loop"))
    full = 160 * 192 * 224
    if op == "pair":
        g = _grid(rng, 24 ** 3, full)
        small = g["D"] * g["H"] * g["W"] < 48 ** 3
        return dict(op="pair", image="blobs" if small else "voronoi", **g, window=5,
                    storage="f32", state="f32", field="f32", **(BLOBS if small else BRAIN))
    if op == "cells":
        return dict(op="pair", image="cells", **_grid(rng, 64 ** 3, 128 * 256 * 256), window=7,
                    storage="bf16", state="bf16", field="f16", **CELLS)
    if op == "sweep":
        pairs, settings = rng.choice(((1, 4), (2, 3), (2, 4), (3, 2), (3, 3)))
        return dict(op="sweep", image="voronoi", **_grid(rng, 64 ** 3, 117 ** 3),
                    pairs=pairs, settings=settings, window=5, storage=rng.choice(("f32", "bf16")),
                    state=rng.choice(("f32", "bf16")), field="f32", **BRAIN)
    if op == "symmetric":
        return dict(op="symmetric", image="voronoi", **_grid(rng, 40 ** 3, 96 * 113 * 101),
                    window=5, **HALF_BRAIN)
    if op == "svf":
        return dict(op="svf", image="voronoi", **_grid(rng, 40 ** 3, full), window=5,
                    steps=rng.choice((5, 6, 7)))
    if op == "adjoint":
        return dict(op="adjoint", image="voronoi", **_grid(rng, 32 ** 3, full),
                    window=rng.choice((3, 5, 7)), fixed_grad=rng.random() < 0.5)
    if op == "lncc":
        return dict(op="lncc", image="voronoi", **_grid(rng, 24 ** 3, full),
                    window=rng.choice((3, 5, 7)), both=rng.random() < 0.5)
    if op == "mi":
        return dict(op="mi", image="voronoi", **_grid(rng, 32 ** 3, full),
                    bins=rng.choice((16, 32, 48, 64)))
    if op == "smooth":
        return dict(op="smooth", **_grid(rng, 24 ** 3, full), channels=rng.choice((1, 3)),
                    sigma=rng.choice((0.5, 1.0, 2.0)))
    if op == "step":
        return dict(op="step", **_grid(rng, 24 ** 3, full), moments=rng.choice(("f32", "bf16")))
    return dict(op="loop", image="voronoi", **_grid(rng, 24 ** 3, 128 ** 3), window=5,
                sigma_grad=rng.choice((0.5, 1.0, 2.0)), sigma_warp=rng.choice((0.5, 1.0)))


# ------------------------------------------------------------------ inputs

def _gen(seed, *k):
    g = torch.Generator(device="cuda")
    s = int(seed)
    for v in k:
        s = (s * 1000003 + v) % (1 << 62)
    g.manual_seed(s)
    return g


def _lowpass(x, sigma):
    """x [..., D, H, W] blurred by a Gaussian in the periodic Fourier domain."""
    f = [torch.fft.fftfreq(n, device=x.device) for n in x.shape[-3:-1]]
    f.append(torch.fft.rfftfreq(x.shape[-1], device=x.device))
    r2 = f[0][:, None, None] ** 2 + f[1][None, :, None] ** 2 + f[2][None, None, :] ** 2
    t = torch.exp(-2.0 * math.pi ** 2 * sigma ** 2 * r2)
    return torch.fft.irfftn(torch.fft.rfftn(x, dim=(-3, -2, -1)) * t, s=x.shape[-3:],
                            dim=(-3, -2, -1))


def _field(shape, sigma, top, gen):
    """A smooth displacement [3, D, H, W] with max |u| = top voxels."""
    u = _lowpass(torch.randn((3,) + shape, device="cuda", generator=gen), sigma)
    return (u * (top / u.square().sum(0).max().sqrt())).contiguous()


def _coords(shape):
    return torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.float32) for n in shape],
                          indexing="ij")


def _pair(image, shape, seed):
    """Fixed and moving image, moving(x) ~ fixed(x + w(x)) for a smooth w."""
    small = min(shape)
    z, y, x = _coords(shape)
    if image == "blobs":
        w = _field(shape, 4.0, 2.0, _gen(seed, 1))
        g = _gen(seed, 2)
        c = torch.rand(8, 3, device="cuda", generator=g) * torch.tensor(shape, device="cuda")
        a = 0.5 + 0.5 * torch.rand(8, device="cuda", generator=g)

        def blobs(z, y, x):
            out = torch.zeros_like(z)
            for k in range(8):
                r2 = (z - c[k, 0]) ** 2 + (y - c[k, 1]) ** 2 + (x - c[k, 2]) ** 2
                out += a[k] * torch.exp(-r2 / 18.0)
            return out
        return blobs(z, y, x), blobs(z + w[0], y + w[1], x + w[2])
    if image == "cells":
        w = _field(shape, 16.0, min(12.0, small / 10.0), _gen(seed, 1))
        g = _gen(seed, 2)
        on = torch.rand(shape, device="cuda", generator=g) < 1e-3
        amp = torch.exp(0.5 * torch.randn(shape, device="cuda", generator=g))
        peak = (2.0 * math.pi * 1.5 ** 2) ** 1.5
        clean = _lowpass(torch.where(on, amp, torch.zeros_like(amp)) * peak, 1.5)
        noise = [0.05 + 0.01 * torch.randn(shape, device="cuda", generator=g) for _ in range(2)]
        return clean + noise[0], _sample(clean[None], w)[0] + noise[1]
    w = _field(shape, 8.0, min(8.0, small / 10.0), _gen(seed, 1))
    g = _gen(seed, 2)
    pts = torch.rand(36, 3, device="cuda", generator=g) * torch.tensor(shape, device="cuda")
    means = 0.1 + 0.9 * torch.rand(36, device="cuda", generator=g)

    def voronoi(z, y, x):
        best = torch.full_like(z, 1e30)
        out = torch.zeros_like(z)
        for k in range(36):
            r2 = (z - pts[k, 0]) ** 2 + (y - pts[k, 1]) ** 2 + (x - pts[k, 2]) ** 2
            near = r2 < best
            best = torch.where(near, r2, best)
            out = torch.where(near, means[k], out)
        out = out + 0.02 * torch.randn(shape, device="cuda", generator=g)
        return _lowpass(out, 1.0)
    return voronoi(z, y, x), voronoi(z + w[0], y + w[1], x + w[2])


_TYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _ints(text):
    return tuple(int(t) for t in text.split(","))


def _params(case, **more):
    return fa.RegParams(scales=_ints(case["scales"]), iters=_ints(case["iters"]),
                        window=case["window"], state=case.get("state", "f32"),
                        field=case.get("field", "f32"), **more)


def _sweep_settings(n):
    return (0.25, 0.5, 1.0, 0.75)[:n]


def _sweep_shapes(case):
    """Uneven grids: the axes of each further pair are a little smaller and permuted."""
    s = (case["D"], case["H"], case["W"])
    return [tuple(max(8, s[(a + k) % 3] - 7 * k) for a in range(3)) for k in range(case["pairs"])]


def prepare(case, seed):
    op = case["op"]
    shape = (case["D"], case["H"], case["W"])
    st = dict(case)
    if op == "sweep":
        two = [_pair(case["image"], s, seed * 31 + k) for k, s in enumerate(_sweep_shapes(case))]
        t = _TYPES[case["storage"]]
        st["fixed"] = [a.to(t).contiguous() for a, _ in two]
        st["moving"] = [b.to(t).contiguous() for _, b in two]
        st["params"] = [_params(case, lr=lr) for lr in _sweep_settings(case["settings"])]
        return st
    if "image" in case:
        a, b = _pair(case["image"], shape, seed)
        t = _TYPES[case.get("storage", "f32")]
        st["fixed"], st["moving"] = a.to(t).contiguous(), b.to(t).contiguous()
    g = _gen(seed, 3)
    if op == "pair":
        st["params"] = _params(case)
    elif op == "symmetric":
        st["params"] = _params(case)
        st["inverse"] = fa.RegParams(scales=(2, 1), iters=(50, 25))
    elif op == "svf":
        st["v"] = _field(shape, 8.0, min(6.0, min(shape) / 12.0), g)
        st["params"] = fa.RegParams(scales=(1,), iters=(0,), window=case["window"])
    elif op == "adjoint":
        st["u"] = _field(shape, 8.0, min(6.0, min(shape) / 12.0), g)
    elif op == "smooth":
        x = torch.randn((case["channels"],) + shape, device="cuda", generator=g)
        st["x"] = (_lowpass(x, 3.0) + 0.1 * x).contiguous()
    elif op in ("step", "loop"):
        # moments as a few iterations of a registration leave them: |g| ~ 1e-7
        t = _TYPES[case.get("moments", "f32")]
        h = 1e-7 * _field(shape, 3.0, 1.0, g)
        noise = 1e-8 * torch.randn(h.shape, device="cuda", generator=g)
        st["u"] = _field(shape, 8.0, min(4.0, min(shape) / 12.0), g)
        st["g"] = (h + noise).contiguous()
        st["m"] = (0.6 * h).to(t).contiguous()
        st["v"] = (0.01 * (h * h + 1e-16)).to(t).contiguous()
        st["t"] = torch.full((1,), 10, dtype=torch.int32, device="cuda")
        st["params"] = fa.RegParams()
    return st


def run(s):
    op = s["op"]
    if op == "pair":
        r = fa.fa_register(s["fixed"], s["moving"], s["params"], sync=False)
        return {"u": r["u"], "loss": r["loss"]}
    if op == "sweep":
        jobs = fa.fa_register_batched_lockstep(s["fixed"], s["moving"], s["params"], sync=False)
        return [{"u": j["u"], "loss": j["loss"]} for j in jobs]
    if op == "symmetric":
        return fa.fa_register_symmetric(s["fixed"], s["moving"], s["params"], s["inverse"],
                                        sync=False)
    if op == "svf":
        loss, g, u = fa.fa_svf_loss_grad(s["fixed"], s["moving"], s["v"], s["steps"], s["params"])
        return {"loss": loss, "grad_v": g, "u": u}
    if op == "adjoint":
        r = fa.fa_warp_lncc_adjoint(s["fixed"], s["moving"], s["u"], window=s["window"],
                                    want_fixed=s["fixed_grad"])
        return {k: v for k, v in r.items() if v is not None}
    if op == "lncc":
        r = fa.fa_lncc_fwd_bwd(s["fixed"], s["moving"], window=s["window"], want_dI=s["both"])
        return {k: v for k, v in r.items() if v is not None}
    if op == "mi":
        return fa.fa_mi_fwd_bwd(s["fixed"], s["moving"], bins=s["bins"])
    if op == "smooth":
        return fa.fa_gauss_smooth(s["x"], s["sigma"])
    if op == "step":
        u, eps = fa.fa_radam_step(s["u"], s["m"], s["v"], s["g"], s["t"], s["params"])
        return {"u": u, "eps": eps, "m": s["m"], "v": s["v"]}
    # one iteration of the registration loop, call by call
    J, grad = fa.fa_warp(s["moving"], s["u"])
    r = fa.fa_lncc_fwd_bwd(s["fixed"], J, window=s["window"])
    g = fa.fa_gauss_smooth(r["dJ"] * grad, s["sigma_grad"])
    u, eps = fa.fa_radam_step(s["u"], s["m"], s["v"], g, s["t"], s["params"])
    return {"u": fa.fa_gauss_smooth(u, s["sigma_warp"]), "loss": r["loss"], "m": s["m"],
            "v": s["v"]}


# ------------------------------------------------------------------ work

def _voxel_iters(shape, case):
    n = 0
    for s, t in zip(_ints(case["scales"]), _ints(case["iters"])):
        n += t * int(np.prod([fa.level_size(a, s) for a in shape]))
    return n


def work(case):
    """Bytes and operations of one pass.  A registration iteration reads the
    two images, u and both moments and writes u and the moments (its state
    does not fit on the chip at the sizes that matter); every other call
    reads its inputs and writes its outputs once.  Operations per voxel count
    the separable sums, filters, interpolations and updates."""
    op = case["op"]
    shape = (case["D"], case["H"], case["W"])
    n = int(np.prod(shape))
    if op in ("pair", "sweep"):
        size = {"f32": 4, "bf16": 2, "f16": 2}
        per = 2 * size[case["storage"]] + 6 * size[case["field"]] + 12 * size[case["state"]]
        shapes = _sweep_shapes(case) * case["settings"] if op == "sweep" else [shape]
        vi = sum(_voxel_iters(s, case) for s in shapes)
        return {"bytes": vi * per, "flops": vi * 350}
    if op == "symmetric":
        vi = _voxel_iters(shape, case)
        inv = _voxel_iters(shape, dict(scales="2,1", iters="50,25"))
        return {"bytes": vi * 152 + inv * 84, "flops": vi * 650 + inv * 300}
    if op == "svf":
        # both images and v in, grad_v and u out; the squarings and their adjoints
        return {"bytes": n * 44, "flops": n * (150 + 200 * case["steps"])}
    if op == "adjoint":
        return {"bytes": n * (4 + 4 + 12 + 12 + 4 + (4 if case["fixed_grad"] else 0)),
                "flops": n * 250}
    if op == "lncc":
        return {"bytes": n * (4 + 4 + 4 + (4 if case["both"] else 0)), "flops": n * 120}
    if op == "mi":
        return {"bytes": n * 12, "flops": n * 140}
    if op == "smooth":
        taps = 2 * math.ceil(3 * case["sigma"]) + 1
        return {"bytes": n * 8 * case["channels"], "flops": n * case["channels"] * 6 * taps}
    if op == "step":
        return {"bytes": n * (36 + 12 * (4 if case["moments"] == "f32" else 2)), "flops": n * 120}
    # loop: both images, u, m, v in; u, m, v out
    return {"bytes": n * 80, "flops": n * 350}


# ------------------------------------------------------------------ 64 bits

def _f32(x):
    return float(np.float32(x))


B1, B2, ADAM_EPS, CC_EPS = _f32(0.9), _f32(0.999), _f32(1e-8), _f32(1e-5)


def _corners(shape, u):
    """The eight corners of the cells of x + u(x): (index, weight, the signs of
    the weight's derivatives with their other factors, inside)."""
    D, H, W = shape
    f = torch.floor(u)
    t = u - f
    base = torch.meshgrid(*[torch.arange(k, device=u.device) for k in u.shape[1:]], indexing="ij")
    i = [b + c.long() for b, c in zip(base, f)]
    for a in range(8):
        bit = (a >> 2 & 1, a >> 1 & 1, a & 1)
        p = [i[k] + bit[k] for k in range(3)]
        w = [t[k] if bit[k] else 1 - t[k] for k in range(3)]
        s = [1.0 if bit[k] else -1.0 for k in range(3)]
        ok = (p[0] >= 0) & (p[0] < D) & (p[1] >= 0) & (p[1] < H) & (p[2] >= 0) & (p[2] < W)
        idx = ((p[0].clamp(0, D - 1) * H + p[1].clamp(0, H - 1)) * W + p[2].clamp(0, W - 1))
        yield idx.reshape(-1), w, s, ok


def _sample(v, u, grad=False):
    """v [C, D, H, W] at x + u(x), trilinear, zero outside; with grad also the
    derivatives [C, 3, ...] inside the cell."""
    C, shape = v.shape[0], tuple(v.shape[1:])
    flat = v.reshape(C, -1)
    out = torch.zeros((C,) + tuple(u.shape[1:]), dtype=v.dtype, device=v.device)
    G = torch.zeros((C, 3) + tuple(u.shape[1:]), dtype=v.dtype, device=v.device) if grad else None
    for idx, w, s, ok in _corners(shape, u):
        val = flat[:, idx].reshape(out.shape) * ok
        out += w[0] * w[1] * w[2] * val
        if grad:
            G[:, 0] += s[0] * w[1] * w[2] * val
            G[:, 1] += s[1] * w[0] * w[2] * val
            G[:, 2] += s[2] * w[0] * w[1] * val
    return (out, G) if grad else out


def _scatter(a, u):
    """The adjoint of _sample in v: a [C, D, H, W] through the cells of x + u(x)."""
    C, shape = a.shape[0], tuple(a.shape[1:])
    out = torch.zeros((C, a[0].numel()), dtype=a.dtype, device=a.device)
    for idx, w, _, ok in _corners(shape, u):
        out.index_add_(1, idx, (a * (w[0] * w[1] * w[2] * ok)).reshape(C, -1))
    return out.reshape(a.shape)


def _slide(x, w, axis):
    """Correlation of x with the taps w along an axis, zero outside."""
    R, n = len(w) // 2, x.shape[axis]
    out = torch.zeros_like(x)
    for k in range(-R, R + 1):
        m = n - abs(k)
        if m > 0:
            out.narrow(axis, max(0, -k), m).add_(x.narrow(axis, max(0, k), m), alpha=w[k + R])
    return out


def _box(x, window):
    for a in (-1, -2, -3):
        x = _slide(x, [1.0] * window, a)
    return x


@functools.lru_cache(maxsize=None)
def _taps(sigma):
    R = math.ceil(3 * sigma)
    w = [math.exp(-k * k / (2 * sigma * sigma)) for k in range(-R, R + 1)]
    return [v / sum(w) for v in w]


def _gauss(x, sigma):
    if sigma == 0:
        return x
    for a in (-1, -2, -3):
        x = _slide(x, _taps(sigma), a)
    return x


def _lncc(I, J, window, want_I=False):
    """Loss, dL/dJ and dL/dI of the squared local correlation."""
    n, N = window ** 3, I.numel()
    sI, sJ = _box(I, window), _box(J, window)
    vI = _box(I * I, window) - sI * sI / n
    vJ = _box(J * J, window) - sJ * sJ / n
    cross = _box(I * J, window) - sI * sJ / n
    den = vI * vJ + CC_EPS
    cc = cross * cross / den

    def side(I, J, sI, sJ, vI):
        A, B = 2 * cross / den, -cc * vI / den
        C = -(A * sI + 2 * B * sJ) / n
        return -(I * _box(A, window) + 2 * J * _box(B, window) + _box(C, window)) / N
    return -cc.mean(), side(I, J, sI, sJ, vI), side(J, I, sJ, sI, vJ) if want_I else None


def _adam(m, v, g, t):
    """Updated moments and the direction of step t."""
    m = B1 * m + (1 - B1) * g
    v = B2 * v + (1 - B2) * g * g
    return m, v, (m / (1 - B1 ** t)) / ((v / (1 - B2 ** t)).sqrt() + ADAM_EPS)


def _eps(d, lr):
    top = float(d.square().sum(0).max().sqrt())
    return lr / (2.0 * top) if top > 0 else 0.0


def _compose(u, delta):
    return delta + _sample(u, delta)


def _resample(v, shape):
    """Trilinear, align-corners."""
    src = v.shape[1:]
    c = []
    for a in range(3):
        k = torch.arange(shape[a], device=v.device, dtype=v.dtype)
        ok = shape[a] > 1 and src[a] > 1
        c.append((k * (src[a] - 1) / (shape[a] - 1) if ok else 0 * k) - k)
    return _sample(v, torch.stack(torch.meshgrid(*c, indexing="ij")))


def _levels(case, shape):
    for s, t in zip(_ints(case["scales"]), _ints(case["iters"])):
        yield s, t, tuple(fa.level_size(a, s) for a in shape)


def _level_image(x, s, shape):
    return x if s == 1 else _resample(_gauss(x, 0.5 * s)[None], shape)[0]


def _handoff(states, shape):
    """u, m, v of each map on the next level's grid."""
    old = states[0][0].shape[1:]
    f = torch.tensor([1.0 if a <= 1 or b <= 1 else (b - 1) / (a - 1) for a, b in zip(old, shape)],
                     dtype=torch.float64, device="cuda").reshape(3, 1, 1, 1)
    return [(_resample(u, shape) * f, _resample(m, shape) / f, _resample(v, shape) / f ** 2)
            for u, m, v in states]


def _update(state, g, t, sigma_grad=1.0, sigma_warp=0.5, lr=0.5):
    u, m, v = state
    m, v, d = _adam(m, v, _gauss(g, sigma_grad), t)
    return _gauss(_compose(u, -_eps(d, lr) * d), sigma_warp), m, v


def _register64(case, fixed, moving, symmetric=False):
    """A registration's final maps and loss; symmetric: both maps move."""
    t, states = 0, None
    for s, iters, shape in _levels(case, fixed.shape):
        If, Im = _level_image(fixed, s, shape), _level_image(moving, s, shape)
        if states is None:
            states = [tuple(torch.zeros((3,) + shape, dtype=torch.float64, device="cuda")
                            for _ in range(3))] * (2 if symmetric else 1)
        else:
            states = _handoff(states, shape)
        for _ in range(iters):
            t += 1
            J, G = _sample(Im[None], states[-1][0], grad=True)
            if symmetric:
                JF, GF = _sample(If[None], states[0][0], grad=True)
                _, dJ, dF = _lncc(JF[0], J[0], case["window"], want_I=True)
                states = [_update(states[0], dF * GF[0], t), _update(states[1], dJ * G[0], t)]
            else:
                _, dJ, _ = _lncc(If, J[0], case["window"])
                states = [_update(states[0], dJ * G[0], t)]
        end = If, Im
    If, Im = end
    if symmetric:
        If = _sample(If[None], states[0][0])[0]
    loss = _lncc(If, _sample(Im[None], states[-1][0])[0], case["window"])[0]
    return [s[0] for s in states], loss


def _svf64(s):
    I, Im, v, steps = (s[k].double() if k != "steps" else s[k]
                       for k in ("fixed", "moving", "v", "steps"))
    us = [v / 2 ** steps]
    for _ in range(steps):
        us.append(_compose(us[-1], us[-1]))
    J, G = _sample(Im[None], us[-1], grad=True)
    loss, dJ, _ = _lncc(I, J[0], s["window"])
    g = dJ * G[0]
    for u in reversed(us[:-1]):
        _, Gu = _sample(u, u, grad=True)
        g = g + torch.einsum("ja...,j...->a...", Gu, g) + _scatter(g, u)
    return {"loss": loss, "grad_v": g / 2 ** steps, "u": us[-1]}


def _spline(t):
    r = 1 - t
    return [r ** 3 / 6, t ** 3 / 2 - t * t + 2 / 3, -t ** 3 / 2 + t * t / 2 + t / 2 + 1 / 6,
            t ** 3 / 6]


def _spline_slope(t):
    r = 1 - t
    return [-r * r / 2, 1.5 * t * t - 2 * t, -1.5 * t * t + t + 0.5, t * t / 2]


def _mi64(I, J, B):
    N = I.numel()

    def place(v, lo, hi):
        x = (1 + (v - lo) * ((B - 3) / (hi - lo))).clamp(1, B - 2).reshape(-1)
        f = torch.floor(x)
        return f.long() - 1, x - f, (B - 3) / (hi - lo)
    a0, ta, _ = place(I, float(I.min()), float(I.max()))
    b0, tb, slope = place(J, min(0.0, float(J.min())), max(0.0, float(J.max())))
    wa, wb, db = _spline(ta), _spline(tb), _spline_slope(tb)
    P = torch.zeros(B * B, dtype=torch.float64, device=I.device)
    key = lambda p, q: ((a0 + p).clamp(max=B - 1) * B + (b0 + q).clamp(max=B - 1))  # noqa: E731
    for p in range(4):
        for q in range(4):
            P += torch.bincount(key(p, q), weights=wa[p] * wb[q], minlength=B * B)
    P = (P / N).reshape(B, B)
    T = torch.where(P > 0, torch.log(P / (P.sum(1, True) * P.sum(0, True))), 0.0)
    acc = sum(T.reshape(-1)[key(p, q)] * wa[p] * db[q] for p in range(4) for q in range(4))
    return {"loss": -(P * T).sum(), "dJ": (-(slope / N) * acc).reshape(I.shape)}


def exact(case, seed):
    op = case["op"]
    if op == "sweep" or "bf16" in (case.get("state"), case.get("storage")):
        return None  # too long, or a result that 16-bit storage decides
    if op in ("pair", "symmetric") and _voxel_iters((case["D"], case["H"], case["W"]),
                                                    case) > 1.5e8:
        return None  # over about 20 seconds
    s = prepare(case, seed)
    if op == "svf":
        return _svf64(s)
    if op == "smooth":
        return _gauss(s["x"].double(), case["sigma"])
    if op == "step":
        m, v, d = _adam(s["m"].double(), s["v"].double(), s["g"].double(), 11)
        e = _eps(d, 0.5)
        stored = case["moments"] == "f32"  # 16-bit moments are what their rounding makes them
        return {"u": _compose(s["u"].double(), -e * d), "eps": torch.tensor(e, dtype=torch.float64),
                "m": m if stored else None, "v": v if stored else None}
    I, J = s["fixed"].double(), s["moving"].double()
    if op == "pair":
        u, loss = _register64(case, I, J)
        return {"u": u[0], "loss": loss}
    if op == "symmetric":  # the final map goes through the inverse, which is not repeated here
        u, mid = _register64(case, I, J, symmetric=True)
        return {"u": None, "uF": u[0], "uM": u[1], "loss": None, "mid_loss": mid}
    if op == "lncc":
        loss, dJ, dI = _lncc(I, J, case["window"], want_I=case["both"])
        return {"loss": loss, "dJ": dJ, "dI": dI} if case["both"] else {"loss": loss, "dJ": dJ}
    if op == "mi":
        return _mi64(I, J, case["bins"])
    u = s["u"].double()
    w, G = _sample(J[None], u, grad=True)
    if op == "adjoint":
        loss, dJ, dI = _lncc(I, w[0], case["window"], want_I=case["fixed_grad"])
        out = {"loss": loss, "dL_du": dJ * G[0], "dL_dmoving": _scatter(dJ[None], u)[0]}
        return dict(out, dL_dfixed=dI) if case["fixed_grad"] else out
    loss, dJ, _ = _lncc(I, w[0], case["window"])
    un, m, v = _update((u, s["m"].double(), s["v"].double()), dJ * G[0], 11,
                       case["sigma_grad"], case["sigma_warp"])
    return {"u": un, "loss": loss, "m": m, "v": v}
