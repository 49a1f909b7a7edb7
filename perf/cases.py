"""The work a user has this library do, as timed and compared cases.

Each case is one call (or the two calls that belong together) of the public
Python binding on inputs a user's program would have in GPU memory.  The kinds:

``project``     A x and H A x of one slice (Algorithm 1, Step 1): the forward model alone, as
                an iterative reconstruction written on top of the library calls it.
``backproject`` A^T s and A^T H s (Step 3), the other half of such a program.
``fan``         Phi~ x = A V^-1 x and Phi~^T s of the fan-beam geometry.
``sinogram``    the measurement-domain steps of an own loop: H z, the Poisson output step, H s.
``tv``          the proximal-TV denoiser as a plug-in.
``denoise``     the learned denoiser on one image or a stack.
``jvp``         the learned denoiser with its directional derivative (a learned iteration's denoiser).
``gradients``   one training pass of the learned denoiser: loss and every gradient.
``solve``       a whole reconstruction of one slice with prox-TV.
``batch``       whole reconstructions of several slices of mixed sizes at once.

The single steps take FP32 buffers; the learned kinds compute in BF16 with
FP32 accumulation.  Sizes are those of the repository's workloads (64^2/30/95,
512^2/64/729, 1024^2/90/1449, the 256/384/512 mix, 512^2/102/736 fan beam, 32
patches of 64^2) and sizes between them.  Whole solves run in FP32 storage with
the damping the 512^2 workload runs with, which keeps a rounding difference
from growing over the iterations; in BF16 storage, or with the network in the
loop, two equally exact runs of a whole solve part by far more than FP32
rounding, so those are measured step by step.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1609_04661_gb300 as dg
from paper_1609_04661_gb300.train_denoiser import load_cnn

DEV = "cuda"
MIX_N = (256, 384, 512)             # image sides, view counts and doses of a mixed queue of scans
MIX_VIEWS = (32, 48, 64, 96, 128)


def listed():
    return [
        # the smallest geometry: the call is a few launches, so launch and host time count
        {"name": "project_64", "kind": "project", "n": 64, "views": 30, "bins": 95},
        # the paper-scale slice: the forward model of one iteration
        {"name": "project_512", "kind": "project", "n": 512, "views": 64, "bins": 729},
        # its transpose
        {"name": "backproject_512", "kind": "backproject", "n": 512, "views": 64, "bins": 729},
        # the largest slice of the workloads
        {"name": "backproject_1024", "kind": "backproject", "n": 1024, "views": 90, "bins": 1449},
        # the scanner's own geometry (flat-detector fan beam, a full rotation)
        {"name": "fan_512", "kind": "fan", "n": 512, "views": 102, "bins": 736},
        # filter and output step of the largest slice
        {"name": "sinogram_1024", "kind": "sinogram", "n": 1024, "views": 90, "bins": 1449},
        # the denoiser alone on an odd size
        {"name": "tv_501", "kind": "tv", "n": 501, "steps": 20},
        # the learned denoiser on the paper-scale slice
        {"name": "denoise_512", "kind": "denoise", "batch": 1, "rows": 512, "cols": 512},
        # a learned iteration's denoiser on a ragged size
        {"name": "jvp_300", "kind": "jvp", "rows": 300, "cols": 300},
        # the training batch
        {"name": "gradients_32x64", "kind": "gradients", "batch": 32, "rows": 64, "cols": 64},
        # the paper-scale reconstruction, all its iterations
        {"name": "solve_512", "kind": "solve", "n": 512, "views": 64, "bins": 729, "iters": 30, "I0": 1e5},
        # a queue of scans of mixed sizes, view counts and doses
        {"name": "batch_12", "kind": "batch", "slices": 12, "iters": 20, "mix": 1},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["project", "project", "backproject", "backproject", "fan", "sinogram", "tv", "tv", "denoise",
                       "denoise", "jvp", "jvp", "gradients", "solve", "solve", "batch"])
    if kind in ("project", "backproject", "sinogram"):
        n = _logint(rng, 64, 1024)
        return {"kind": kind, "n": n, "views": rng.randint(16, 90), "bins": math.ceil(1.42 * n) + rng.randint(-9, 9)}
    if kind == "fan":
        n = _logint(rng, 64, 400)
        return {"kind": kind, "n": n, "views": rng.randint(24, 96), "bins": math.ceil(1.44 * n)}
    if kind == "tv":
        return {"kind": kind, "n": _logint(rng, 64, 1024), "steps": rng.choice([10, 20, 20, 30])}
    if kind == "denoise":
        return {"kind": kind, "batch": rng.choice([1, 1, 2, 3]), "rows": _logint(rng, 48, 400), "cols": _logint(rng, 48, 400)}
    if kind == "jvp":
        return {"kind": kind, "rows": _logint(rng, 64, 512), "cols": _logint(rng, 64, 512)}
    if kind == "gradients":
        return {"kind": kind, "batch": rng.randint(4, 32), "rows": rng.randint(40, 64), "cols": rng.randint(40, 80)}
    if kind == "solve":
        n = _logint(rng, 64, 512)
        return {"kind": kind, "n": n, "views": max(24, int(n * rng.uniform(0.12, 0.3))), "bins": math.ceil(1.42 * n),
                "iters": rng.randint(5, 30), "I0": 10.0 ** rng.uniform(4, 6)}
    return {"kind": kind, "slices": rng.randint(3, 11), "iters": rng.randint(5, 20), "mix": rng.randrange(1 << 30)}


# ---------------------------------------------------------------- inputs ----
def _ellipses(n, seed, count=10):
    """Random ellipses inside the field of view: (centre, semi-axes, rotation, density)."""
    g = np.random.default_rng(seed)
    half, out = n / 2.0, []
    for _ in range(count):
        rad, ang = 0.6 * half * math.sqrt(g.uniform()), g.uniform(0, 2 * math.pi)
        a, b = g.uniform(0.05, 0.4, 2) * half
        out.append((rad * math.cos(ang), rad * math.sin(ang), a, b, g.uniform(0, math.pi),
                    g.uniform(0, 0.02) * min(1.0, 512.0 / n)))
    return out


def _image(n, seed):
    """Attenuation map [n][n] (float32, GPU)."""
    c = (n - 1) / 2.0
    k = torch.arange(n, device=DEV, dtype=torch.float32)
    X, Y = (k - c)[None, :], (c - k)[:, None]
    img = torch.zeros((n, n), device=DEV)
    for x0, y0, a, b, phi, rho in _ellipses(n, seed):
        u = math.cos(phi) * (X - x0) + math.sin(phi) * (Y - y0)
        v = -math.sin(phi) * (X - x0) + math.cos(phi) * (Y - y0)
        img += rho * ((u / a) ** 2 + (v / b) ** 2 <= 1.0)
    return img


def _lines(n, views, bins, seed):
    """The ellipses' line integrals [views][bins] (float64, GPU): parallel beam, half a turn."""
    th = (torch.arange(views, device=DEV, dtype=torch.float64) * (math.pi / views))[:, None]
    u = (torch.arange(bins, device=DEV, dtype=torch.float64) - (bins - 1) / 2.0)[None, :]
    z = torch.zeros((views, bins), device=DEV, dtype=torch.float64)
    for x0, y0, a, b, phi, rho in _ellipses(n, seed):
        q = a * a * torch.cos(th - phi) ** 2 + b * b * torch.sin(th - phi) ** 2
        t = u - x0 * torch.cos(th) - y0 * torch.sin(th)
        z += 2 * rho * a * b * torch.sqrt(torch.clamp(q - t * t, min=0.0)) / q
    return z


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _counts(z, I0, seed):
    return torch.poisson(I0 * torch.exp(-z), generator=_gen(seed)).float()


def _residual(n, views, bins, seed):
    """What a back-projection is given: the data's misfit, signed and noisy."""
    z = _lines(n, views, bins, seed)
    return (0.1 * (z - z.mean()) + 0.05 * torch.randn(z.shape, generator=_gen(seed), device=DEV)).float().contiguous()


def _fan(case):
    n = case["n"]       # a clinical scanner's proportions
    return dict(src_dist=900.0 / 512 * n, det_dist=740.0 / 512 * n, det_spacing=1.95)


def _mix(case, seed):
    """Sizes (from the case alone) and seeds of a batch's slices."""
    g = np.random.default_rng(case["mix"])
    out = []
    for k in range(case["slices"]):
        n, v = int(g.choice(MIX_N)), int(g.choice(MIX_VIEWS))
        out.append((n, v, math.ceil(1.42 * n), float(10.0 ** g.uniform(4, 6)), 1000 * seed + k))
    return out


def _noisy(shape, seed, lo=0.02, hi=0.3):
    """Noisy images [B][H][W], the clean ones and their noise levels."""
    B, H, W = shape
    m = max(H, W)
    x = torch.stack([20.0 * _image(m, 1000 * seed + k)[:H, :W] for k in range(B)])
    s = np.exp(np.random.default_rng(seed).uniform(math.log(lo), math.log(hi), B)).astype(np.float32)
    r = x + torch.as_tensor(s, device=DEV)[:, None, None] * torch.randn(shape, generator=_gen(seed), device=DEV)
    return r.contiguous(), x.contiguous(), s


SOLVE = dict(c_tv=3.0, k_tv=20, damp_x=0.2, damp_s=0.15)


def _inputs(case, seed):
    """The tensors (and numbers) of a case, without plan or network."""
    k = case["kind"]
    if k == "project":
        n = case["n"]
        return {"x": (_image(n, seed) + 0.002 * torch.randn((n, n), generator=_gen(seed), device=DEV)).contiguous()}
    if k == "backproject":
        return {"s": _residual(case["n"], case["views"], case["bins"], seed)}
    if k == "fan":
        n = case["n"]
        return {"x": (_image(n, seed) + 0.002 * torch.randn((n, n), generator=_gen(seed), device=DEV)).contiguous(),
                "s": _residual(n, case["views"], case["bins"], seed)}
    if k == "sinogram":
        z = _lines(case["n"], case["views"], case["bins"], seed)
        e = torch.randn(z.shape, generator=_gen(seed + 1), device=DEV)
        return {"raw": z.float().contiguous(), "z": (z + 0.05 * e).float().contiguous(),
                "y": _counts(z, 1e5, seed).contiguous(), "s0": (0.3 * e).contiguous(), "I0": 1e5, "tau_p": 0.02}
    if k == "tv":
        n = case["n"]
        x = 20.0 * _image(n, seed)
        return {"r": (x + 0.05 * torch.randn((n, n), generator=_gen(seed), device=DEV)).contiguous(), "lam": 0.15}
    if k == "denoise":
        r, _, s = _noisy((case["batch"], case["rows"], case["cols"]), seed)
        return {"r": r, "sigma": s}
    if k == "jvp":
        r, _, s = _noisy((1, case["rows"], case["cols"]), seed)
        b = torch.randn(r.shape[1:], generator=_gen(seed + 7), device=DEV)
        return {"r": r[0].contiguous(), "b": b.contiguous(), "sigma": float(s[0])}
    if k == "gradients":
        r, x, s = _noisy((case["batch"], case["rows"], case["cols"]), seed)
        return {"r": r, "x": x, "sigma": s}
    if k == "solve":
        return {"y": _counts(_lines(case["n"], case["views"], case["bins"], seed), case["I0"], seed).contiguous()}
    return {"y": [_counts(_lines(n, v, d, sd), I0, sd).contiguous() for n, v, d, I0, sd in _mix(case, seed)],
            "I0": [m[3] for m in _mix(case, seed)]}


def prepare(case, seed):
    k, st = case["kind"], {"case": case}
    if k in ("denoise", "jvp", "gradients"):
        st["net"] = load_cnn()
    elif k == "batch":
        st["plans"] = [dg.Plan(n, v, d, **SOLVE) for n, v, d, _, _ in _mix(case, seed)]
        st["batch"] = dg.Batch(st["plans"])
    elif k == "tv":
        st["plan"] = dg.Plan(case["n"], 32, math.ceil(1.42 * case["n"]), k_tv=case["steps"])
    elif k == "fan":
        st["plan"] = dg.Plan(case["n"], case["views"], case["bins"], fan=_fan(case))
    else:
        st["plan"] = dg.Plan(case["n"], case["views"], case["bins"], **(SOLVE if k == "solve" else {}))
    st.update(_inputs(case, seed))
    return st


def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "project":
        return st["plan"].project(st["x"]), st["plan"].project(st["x"], precond=True)
    if k == "backproject":
        return st["plan"].backproject(st["s"]), st["plan"].backproject(st["s"], precond=True)
    if k == "fan":
        return st["plan"].project(st["x"], precond=True), st["plan"].backproject(st["s"], precond=True)
    if k == "sinogram":
        s, tau_s = st["plan"].output_step(st["z"], st["y"], st["s0"], st["I0"], st["tau_p"])
        return st["plan"].filter(st["raw"]), s, tau_s, st["plan"].filter(st["s0"])
    if k == "tv":
        return st["plan"].denoise_tv(st["r"], st["lam"])
    if k == "denoise":
        return st["net"].denoise(st["r"], st["sigma"])
    if k == "jvp":
        return st["net"].denoise_jvp(st["r"], st["b"], st["sigma"])
    if k == "gradients":
        return st["net"].gradients(st["r"], st["x"], st["sigma"])
    if k == "solve":
        return st["plan"].solve(st["y"], case["I0"], case["iters"])
    return st["batch"].solve(st["y"], st["I0"], case["iters"])


# ------------------------------------------------------------------ work ----
CNN_MACS = 15 * 9 * 64 * 64 + 2 * 9 * 64       # multiply-adds per pixel of the 17-layer network
TV_FLOPS = 19                                  # per pixel and step: divergence, gradient, its length, projection


def _solve_work(n, views, bins, iters):
    """Counts in, image out; per iteration A and A^T (two taps a step), H twice (one padded FFT pair each),
    the output step and 20 TV steps on the pair of images that the divergence takes."""
    P = 1 << (2 * bins - 1).bit_length()
    fft = 2 * 5 * P * math.log2(P)
    it = 2 * 4 * views * bins * n + 2 * views * fft + 30 * views * bins + 2 * 20 * TV_FLOPS * n * n
    return 4 * (views * bins + n * n), iters * it


def work(case):
    k = case["kind"]
    if k in ("project", "backproject", "fan", "sinogram"):
        n, M, N = case["n"], case["views"] * case["bins"], case["n"] ** 2
        P = 1 << (2 * case["bins"] - 1).bit_length()
        H = case["views"] * 2 * 5 * P * math.log2(P)
        if k in ("project", "backproject"):
            one = N + 2 * M if k == "project" else M + 2 * N
            return {"bytes": 4 * one, "flops": 2 * 4 * M * n + H}
        if k == "fan":
            m = 1 << (2 * n - 1).bit_length()
            return {"bytes": 4 * 2 * (M + N), "flops": 2 * 4 * M * n + 2 * 2 * 5 * m * m * math.log2(m * m)}
        return {"bytes": 4 * 7 * M, "flops": 2 * H + 30 * M}
    if k == "tv":
        return {"bytes": 8 * case["n"] ** 2, "flops": TV_FLOPS * case["steps"] * case["n"] ** 2}
    if k in ("denoise", "jvp", "gradients"):
        pix = case.get("batch", 1) * case["rows"] * case["cols"]
        passes = {"denoise": 1, "jvp": 2, "gradients": 3}[k]
        weights = 2 * CNN_MACS
        return {"bytes": 4 * pix * {"denoise": 2, "jvp": 4, "gradients": 2}[k] + weights * (3 if k == "gradients" else 1),
                "flops": 2.0 * CNN_MACS * pix * passes}
    if k == "solve":
        b, f = _solve_work(case["n"], case["views"], case["bins"], case["iters"])
        return {"bytes": b, "flops": f}
    w = [_solve_work(n, v, d, case["iters"]) for n, v, d, _, _ in _mix(case, 0)]
    return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}


# ---------------------------------------------------------- 64-bit values ----
def _parallel_rays(n, views, bins, k):
    """Joseph's method for view k: (fractional index across the march [bins][n], by columns?, step length)."""
    th, c = k * math.pi / views, (n - 1) / 2.0
    u = (torch.arange(bins, device=DEV, dtype=torch.float64) - (bins - 1) / 2.0)[:, None]
    q = torch.arange(n, device=DEV, dtype=torch.float64)[None, :] - c
    s, t = math.sin(th), math.cos(th)
    if abs(s) >= abs(t):
        return c - (u - q * t) / s, torch.ones(bins, 1, dtype=torch.bool, device=DEV), torch.full((bins, 1), 1 / abs(s), device=DEV, dtype=torch.float64)
    return (u + q * s) / t + c, torch.zeros(bins, 1, dtype=torch.bool, device=DEV), torch.full((bins, 1), 1 / abs(t), device=DEV, dtype=torch.float64)


def _fan_rays(n, views, bins, k, fan):
    th, c = k * 2 * math.pi / views, (n - 1) / 2.0
    s, t = math.sin(th), math.cos(th)
    u = (torch.arange(bins, device=DEV, dtype=torch.float64) - (bins - 1) / 2.0)[:, None] * fan["det_spacing"]
    sx, sy = fan["src_dist"] * s, -fan["src_dist"] * t
    vx, vy = -fan["det_dist"] * s + u * t - sx, fan["det_dist"] * t + u * s - sy
    q = torch.arange(n, device=DEV, dtype=torch.float64)[None, :] - c
    col = vx.abs() >= vy.abs()
    pos = torch.where(col, c - (sy + (q - sx) * vy / vx), sx + (-q - sy) * vx / vy + c)
    L = torch.sqrt(vx * vx + vy * vy)
    return pos, col, L / torch.where(col, vx.abs(), vy.abs())


def _taps(n, pos, col, w):
    """Pixel indices and weights [2][bins][n] of the two taps of every step."""
    i0 = torch.floor(pos)
    f = pos - i0
    idx = torch.stack([i0, i0 + 1]).long()
    wt = torch.stack([(1 - f) * w, f * w])
    ok = (idx >= 0) & (idx < n)
    q = torch.arange(n, device=DEV)[None, None, :].expand_as(idx)
    flat = torch.where(col[None], idx * n + q, q * n + idx)
    return torch.where(ok, flat, torch.zeros_like(flat)), torch.where(ok, wt, torch.zeros_like(wt))


def _A(x, case, rays):
    n, flat = case["n"], x.double().reshape(-1)
    out = []
    for k in range(case["views"]):
        idx, wt = _taps(n, *rays(k))
        out.append((flat[idx] * wt).sum((0, 2)))
    return torch.stack(out)


def _At(s, case, rays):
    n = case["n"]
    acc = torch.zeros(n * n, device=DEV, dtype=torch.float64)
    for k in range(case["views"]):
        idx, wt = _taps(n, *rays(k))
        acc.index_add_(0, idx.reshape(-1), (wt * s[k].double()[None, :, None]).reshape(-1))
    return acc.reshape(n, n)


def _floor(bins):
    P = 1 << (2 * bins - 1).bit_length()
    return P, 1.0 / (2 * P)


def _H(z):
    """sqrt(max(|f|, 1/(2P))) along the detector, zero-padded to P."""
    P, f0 = _floor(z.shape[1])
    g = torch.fft.fftfreq(P, device=DEV, dtype=torch.float64).abs().clamp(min=f0).sqrt()
    return torch.fft.ifft(torch.fft.fft(z.double(), n=P, dim=1) * g, dim=1).real[:, :z.shape[1]].contiguous()


def _Vinv(x, bins):
    n = x.shape[0]
    m, f0 = 1 << (2 * n - 1).bit_length(), _floor(bins)[1]
    f = torch.fft.fftfreq(m, device=DEV, dtype=torch.float64)
    g = torch.sqrt(f[:, None] ** 2 + f[None, :] ** 2).clamp(min=f0).sqrt()
    return torch.fft.ifft2(torch.fft.fft2(x.double(), s=(m, m)) * g).real[:n, :n].contiguous()


def _output_step(z, y, s0, I0, tau):
    """Mode of N(z; p, tau) Poisson(y; I0 e^-z) by bisection: s and the mean curvature term."""
    p, y = z.double() - tau * s0.double(), y.double()
    # the root lies between p and log(I0 / y); without counts it is above p by the Lambert-W bound
    L = torch.where(y > 0, torch.log(I0 / y.clamp(min=1.0)), p + torch.log1p(tau * I0 * torch.exp(-p)))
    lo, hi = torch.minimum(p, L), torch.maximum(p, L)
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        up = (mid - p) / tau + y - I0 * torch.exp(-mid) < 0
        lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
    z0 = 0.5 * (lo + hi)
    w = I0 * torch.exp(-z0)
    return (z0 - p) / tau, (w / (1 + tau * w)).mean().reshape(1)


def _tv(r, lam, steps):
    """Chambolle's projection, 1/8 steps from zero."""
    r = r.double()
    px, py = torch.zeros_like(r), torch.zeros_like(r)

    def div():
        d = torch.zeros_like(r)
        d[:, :-1] += px[:, :-1]
        d[:, 1:] -= px[:, :-1]
        d[:-1] += py[:-1]
        d[1:] -= py[:-1]
        return d

    for _ in range(steps):
        q = div() - r / lam
        gx, gy = torch.zeros_like(r), torch.zeros_like(r)
        gx[:, :-1] = q[:, 1:] - q[:, :-1]
        gy[:-1] = q[1:] - q[:-1]
        den = 1 + torch.sqrt(gx * gx + gy * gy) / 8
        px, py = (px + gx / 8) / den, (py + gy / 8) / den
    return r - lam * div()


def _weights():
    """The shipped network's weights as the layers use them (rounded to BF16), and its biases, flat views in 64 bits."""
    net = load_cnn()
    flat = torch.as_tensor(net.get_params(), device=DEV)
    L, out, o = net.layers, [], 0
    for l in range(L):
        ci, co = 1 if l == 0 else 64, 1 if l == L - 1 else 64
        w = flat[o:o + 9 * ci * co].bfloat16().double().reshape(3, 3, ci, co)
        b = flat[o + 9 * ci * co:o + 9 * ci * co + co].double()
        out.append((w, b))
        o += 9 * ci * co + co
    return out


def _net(u, params):
    a = u[:, None]
    for l, (w, b) in enumerate(params):
        a = torch.nn.functional.conv2d(a, w.permute(3, 2, 0, 1), b, padding=1)
        if l < len(params) - 1:
            a = torch.relu(a)
    return a[:, 0]


def exact(case, seed):
    k = case["kind"]
    if k in ("solve", "batch"):
        return None         # no closed form: an iteration of many steps, compared with another run of it
    i = _inputs(case, seed)
    if k in ("project", "backproject"):
        def rays(v):
            return _parallel_rays(case["n"], case["views"], case["bins"], v)
        if k == "project":
            z = _A(i["x"], case, rays)
            return z, _H(z)
        return _At(i["s"], case, rays), _At(_H(i["s"]), case, rays)
    if k == "fan":
        def rays(v):
            return _fan_rays(case["n"], case["views"], case["bins"], v, _fan(case))
        return _A(_Vinv(i["x"], case["bins"]), case, rays), _Vinv(_At(i["s"], case, rays), case["bins"])
    if k == "sinogram":
        s, tau_s = _output_step(i["z"], i["y"], i["s0"], i["I0"], i["tau_p"])
        return _H(i["raw"]), s, tau_s, _H(i["s0"])
    if k == "tv":
        return _tv(i["r"], i["lam"], case["steps"])
    params = _weights()
    with torch.no_grad():
        if k == "denoise":
            s = torch.as_tensor(i["sigma"], device=DEV).double()[:, None, None]
            r = i["r"].double()
            return r - s * _net(r / s, params)
        if k == "jvp":
            s, r, b = i["sigma"], i["r"].double()[None], i["b"].double()[None]
            f, t = torch.func.jvp(lambda u: _net(u, params), (r / s,), (b / s,))
            return (r - s * f)[0], (b - s * t)[0]
    s = torch.as_tensor(i["sigma"], device=DEV).double()[:, None, None]
    r, x = i["r"].double(), i["x"].double()
    leaves = [t.clone().requires_grad_() for wb in params for t in wb]
    f = _net(r / s, [(leaves[2 * l], leaves[2 * l + 1]) for l in range(len(params))])
    loss = (((r - s * f - x) / s) ** 2).mean()
    grads = torch.autograd.grad(loss, leaves)
    return float(loss.detach()), torch.cat([g.reshape(-1) for g in grads]).cpu().numpy()
