"""The measured work of the framework: whole restorations (one image, a batch, a served
stream, a volume) and the operations a program composes itself (one level's solve, its
start, one application of H), through the public binding.

Inputs are seeded synthetic images as in the tests and the benchmark: piecewise-constant
shapes plus a linear gradient on the [0, 255] grey scale, blurred with the case's PSF (zero
boundary) and Gaussian noise of a relative level v; the plan gets the noise's RMS as its
stopping level, as a user who knows the noise gives it.  `exact` is the method in plain
64-bit torch.
"""
import math

import numpy as np
import torch

from paper_2311_03010_gb300 import eecmg as E
from paper_2311_03010_gb300 import synth

TAU, KPM = 0.2, 10.0  # the binding's defaults: Perona-Malik step and contrast


# ------------------------------------------------------------------ the cases


def listed():
    return [
        # The smallest image in use: launches and barriers count.
        {"name": "restore_64", "kind": "restore", "h": 64, "w": 64, "levels": 3, "psf": "gauss", "sigma": 1.5, "band": 4, "v": 0.01,
         "smoother": "mr2", "storage": "fp32"},
        # An ordinary photograph-sized tile through the per-image call.
        {"name": "restore_512", "kind": "restore", "h": 512, "w": 512, "levels": 5, "psf": "gauss", "sigma": 2.5, "band": 7, "v": 0.01,
         "smoother": "mr2", "storage": "fp32"},
        # Ragged sides, motion blur (no separable factors), BF16 search directions.
        {"name": "restore_motion_bf16", "kind": "restore", "h": 1537, "w": 2047, "levels": 5, "psf": "motion", "length": 15, "angle": 30.0,
         "v": 0.01, "smoother": "mr2", "storage": "bf16"},
        # The benchmark's headline: one 4096^2 image through the batched call.
        {"name": "batch_4096", "kind": "batch", "n": 1, "smin": 4096, "smax": 4096, "levels": 5, "psf": "gauss", "sigma": 3.0, "band": 10,
         "v": 0.01, "pick": 0},
        # Many images of uneven sizes, PSFs and noise in one call.
        {"name": "batch_uneven", "kind": "batch", "n": 24, "smin": 128, "smax": 1536, "levels": 5, "psf": "mix", "v": 0.0, "pick": 7},
        # A burst of requests through the server.
        {"name": "serve_mixed", "kind": "serve", "n": 24, "smin": 256, "smax": 2048, "levels": 5, "psf": "mix", "v": 0.0, "pick": 3},
        # One level's solver on its own: CGLS with a motion blur and a fixed count.
        {"name": "solve_cgls_motion", "kind": "solve", "h": 1024, "w": 1024, "levels": 3, "psf": "motion", "length": 11, "angle": 60.0,
         "v": 0.02, "smoother": "cgls", "storage": "fp32", "m": 4},
        # The start of a large prolonged level: extrapolation, interpolation, smoothing, denoising.
        {"name": "start_4096", "kind": "start", "h": 4096, "w": 4096, "levels": 3, "psf": "gauss", "sigma": 3.0, "band": 10, "v": 0.01},
        # The blur alone, as a program that simulates data or computes residuals applies it.
        {"name": "apply_gauss", "kind": "apply", "h": 2160, "w": 3840, "levels": 1, "psf": "gauss", "sigma": 2.0, "band": 6, "v": 0.01,
         "transpose": False},
        # The volume workload of the benchmark.
        {"name": "vol_restore_256", "kind": "vol_restore", "d": 256, "h": 256, "w": 256, "levels": 4, "psf": "gauss3", "sigma": 1.5, "band": 3,
         "v": 0.01},
        # A small ragged volume, where launches and barriers count.
        {"name": "vol_restore_small", "kind": "vol_restore", "d": 45, "h": 70, "w": 61, "levels": 3, "psf": "gauss3", "sigma": 1.0, "band": 2,
         "v": 0.02},
        # One level's solver on a volume with a PSF that has no separable factors.
        {"name": "vol_solve_oblique", "kind": "vol_solve", "d": 96, "h": 121, "w": 150, "levels": 2, "psf": "oblique3", "sigma": 0.8, "band": 2,
         "v": 0.01, "m": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["restore", "restore", "batch", "serve", "solve", "start", "apply", "vol_restore", "vol_solve", "vol_start"])
    c = {"kind": kind}
    if kind in ("batch", "serve"):
        lo = _log_int(rng, 128, 400)
        c |= {"pick": rng.randrange(1 << 20), "n": rng.randint(2, 20), "smin": lo, "smax": lo + _log_int(rng, 64, 1000), "levels": rng.randint(3, 5), "psf": "mix", "v": 0.0}
        return c
    c["v"] = round(rng.uniform(0.005, 0.05), 4)
    if kind.startswith("vol"):
        c |= {"d": _log_int(rng, 24, 160), "h": _log_int(rng, 24, 200), "w": _log_int(rng, 24, 200), "levels": 3}
        if kind != "vol_start" and rng.random() < 0.3:
            c |= {"psf": "oblique3", "sigma": round(rng.uniform(0.6, 1.0), 3), "band": rng.randint(1, 2)}
        else:
            s = round(rng.uniform(0.6, 1.9), 3)
            c |= {"psf": "gauss3", "sigma": s, "band": min(6, math.ceil(3 * s))}
        if kind == "vol_solve":
            c["m"] = rng.randint(1, 4)
        return c
    big = 2400 if kind in ("restore", "solve") else 3800
    c |= {"h": _log_int(rng, 48, big), "w": _log_int(rng, 48, big), "levels": rng.randint(3, 5)}
    if rng.random() < 0.5:
        s = round(rng.uniform(1.0, 4.0), 3)
        c |= {"psf": "gauss", "sigma": s, "band": math.ceil(3 * s)}
    else:
        c |= {"psf": "motion", "length": rng.randint(5, 21), "angle": round(rng.uniform(0.0, 180.0), 1)}
    if kind in ("restore", "solve"):
        c |= {"smoother": rng.choice(["mr2", "mr2", "cgls"]), "storage": rng.choice(["fp32", "fp32", "bf16"])}
    if kind == "solve":
        c["m"] = rng.randint(1, 5)
    if kind == "apply":
        c["transpose"] = rng.random() < 0.5
    return c


# ------------------------------------------------------------------ inputs


def _psf(c):
    """The case's PSF, FP64, odd sides."""
    if c["psf"] == "gauss":
        return synth.gaussian_psf(c["sigma"], c["band"])
    if c["psf"] == "motion":
        return synth.motion_psf(c["length"], c["angle"])
    if c["psf"] == "gauss3":
        return synth.gaussian_psf3(c["sigma"], c["band"])
    i = np.arange(-c["band"], c["band"] + 1, dtype=np.float64)
    z, y, x = np.meshgrid(i, i, i, indexing="ij")
    k = np.exp(-(z * z + y * y + x * x + 0.9 * x * y + 0.5 * y * z) / (2.0 * c["sigma"] ** 2))
    return k / k.sum()


def _shape(c):
    return (c["d"], c["h"], c["w"]) if "d" in c else (c["h"], c["w"])


def _clean(shape, rng):
    """A piecewise-constant image or volume with a linear gradient, on the GPU."""
    dev = "cuda"
    axes = [torch.arange(n, device=dev, dtype=torch.float32).reshape([-1 if j == i else 1 for j in range(len(shape))])
            for i, n in enumerate(shape)]
    n = 1
    for s in shape:
        n *= s
    img = torch.full(shape, float(rng.uniform(0, 255)), device=dev)
    for i in range(min(24, 8 + n // (1 << 18))):
        lo, hi = [], []
        for s in shape:
            r, m = 0.5 * rng.uniform(0.05, 0.40) * s, rng.uniform(0, s)
            lo.append(max(0, int(m - r)))
            hi.append(min(s, int(m + r) + 1))
        val = float(rng.uniform(0, 255))
        part = img[tuple(slice(a, b) for a, b in zip(lo, hi))]
        if i % 2 == 0:
            part.fill_(val)
        elif part.numel():
            d2 = sum(((ax.narrow(j, lo[j], hi[j] - lo[j]) - 0.5 * (lo[j] + hi[j] - 1)) / max(0.5, 0.5 * (hi[j] - lo[j]))) ** 2
                     for j, ax in enumerate(axes))
            part.masked_fill_(d2 <= 1.0, val)
    swing, way = rng.uniform(20.0, 60.0), rng.standard_normal(len(shape))
    way /= np.linalg.norm(way)
    span = sum(abs(a) * max(s - 1, 1) for a, s in zip(way, shape))
    for a, ax, s in zip(way, axes, shape):
        img += (ax - 0.5 * (s - 1)) * float(a * swing / span)
    return img.clamp_(0.0, 255.0)


def _degraded(shape, psf, v, seed):
    """(clean image, its blurred and noisy data, the noise's RMS), FP32."""
    rng = np.random.default_rng(seed)
    u = _clean(shape, rng)
    full = [a + b - 1 for a, b in zip(shape, psf.shape)]
    fast = [s + (-s) % 16 for s in full]
    f = torch.fft.rfftn(u.double(), s=fast) * torch.fft.rfftn(torch.as_tensor(psf, device="cuda"), s=fast)
    b = torch.fft.irfftn(f, s=fast)[tuple(slice(k // 2, k // 2 + s) for k, s in zip(psf.shape, shape))]
    gen = torch.Generator("cuda").manual_seed(seed)
    e = torch.randn(shape, device="cuda", generator=gen)
    e *= v * float(u.norm()) / float(e.norm())
    return u, (b + e).float().contiguous(), float(e.double().square().mean().sqrt())


def _items(c, seed):
    """The images of a batch or of a burst: sizes, PSFs and noise from the case (the same for
    every seed, as a program's plans are), pixels from the seed."""
    rng = np.random.default_rng(1000 + c["pick"])
    got = []
    for i in range(c["n"]):
        s = int(round(math.exp(rng.uniform(math.log(c["smin"]), math.log(c["smax"]))))) if c["kind"] == "serve" else int(rng.integers(c["smin"], c["smax"] + 1))
        h = w = s
        if c["n"] > 1 and rng.uniform() < 0.5:
            h, w = (s, max(32, round(0.75 * s)))[::1 if rng.uniform() < 0.5 else -1]
        d = {"h": h, "w": w, "levels": c["levels"], "smoother": "mr2", "storage": "fp32"}
        if c["psf"] == "mix":
            if rng.uniform() < 0.5:
                sig = float(rng.uniform(1.0, 4.0))
                d |= {"psf": "gauss", "sigma": sig, "band": math.ceil(3 * sig)}
            else:
                d |= {"psf": "motion", "length": int(rng.integers(5, 22)), "angle": float(rng.uniform(0.0, 180.0))}
            d["v"] = float(rng.uniform(0.005, 0.05))
        else:
            d |= {"psf": c["psf"], "sigma": c["sigma"], "band": c["band"], "v": c["v"]}
        got.append((d, seed + 7919 * i))
    return got


def _start_inputs(c, seed):
    """Two coarser levels' solutions as a cascade meets them: near-equal where they share pixels."""
    _, g, _ = _degraded(_shape(c), np.ones((1,) * len(_shape(c))), c["v"], seed)
    half, quarter = (slice(None, None, 2),) * g.dim(), (slice(None, None, 4),) * g.dim()
    u2 = g[quarter].contiguous()
    u2 += 0.5 * torch.randn(u2.shape, device="cuda", generator=torch.Generator("cuda").manual_seed(seed + 1))
    return g[half].contiguous(), u2


def _plan(c, delta, **kw):
    return E.Plan(c["w"], c["h"], c["levels"], _psf(c), TAU, KPM, smoother=c.get("smoother", "cgls"), storage=c.get("storage", "fp32"),
                  delta=delta, **kw)


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("batch", "serve"):
        plans, gs, us = [], [], []
        for d, s in _items(c, seed):
            _, g, delta = _degraded(_shape(d), _psf(d), d["v"], s)
            plans.append(_plan(d, delta, workspace=0 if kind == "serve" else 1))
            gs.append(g)
            us.append(torch.empty_like(g))
        st = {"kind": kind, "plans": plans, "g": gs, "u": us}
        if kind == "serve":
            st["server"] = E.Server(6 << 30, 64)
        return st
    if kind in ("start", "vol_start"):
        u1, u2 = _start_inputs(c, seed)
        plan = E.VolumePlan(c["w"], c["h"], c["d"], c["levels"], _psf(c), TAU, KPM, delta=1.0) if "d" in c else _plan(c, 1.0)
        return {"kind": kind, "plan": plan, "level": c["levels"] - 1, "u1": u1, "u2": u2, "u": torch.empty(_shape(c), device="cuda")}
    clean, g, delta = _degraded(_shape(c), _psf(c), c["v"], seed)
    if kind == "apply":
        return {"kind": kind, "plan": _plan(c, 1.0), "level": c["levels"] - 1, "x": clean, "u": torch.empty_like(g), "transpose": int(c["transpose"])}
    # a solver on its own runs the count it is given; a restoration stops at the noise
    stop = {"stop": "fixed"} if kind.endswith("solve") else {}
    if "d" in c:
        plan = E.VolumePlan(c["w"], c["h"], c["d"], c["levels"], _psf(c), TAU, KPM, delta=delta, **stop)
    else:
        plan = _plan(c, delta, **stop)
    return {"kind": kind, "plan": plan, "level": c["levels"] - 1, "m": c.get("m", 0), "g": g, "u": torch.empty_like(g)}


def run(s):
    kind = s["kind"]
    if kind == "restore" or kind == "vol_restore":
        s["plan"].restore(s["g"], s["u"])
    elif kind == "batch":
        E.eecmg_restore_batched([p.handle for p in s["plans"]], s["g"], s["u"])
    elif kind == "serve":
        for p, g, u in zip(s["plans"], s["g"], s["u"]):
            s["server"].submit(p, g, u)
        s["server"].drain()
    elif kind == "solve":  # in place, from the data as the start
        s["u"].copy_(s["g"])
        E.eecmg_level_solve(s["plan"].handle, s["level"], s["g"], s["u"], s["m"])
    elif kind == "vol_solve":
        s["u"].copy_(s["g"])
        E.eecmg_vol_level_solve(s["plan"].h, s["level"], s["g"], s["u"], s["m"])
    elif kind == "start":
        E.eecmg_start_level(s["plan"].handle, s["level"], s["u1"], s["u2"], s["u"])
    elif kind == "vol_start":
        E.eecmg_vol_start_level(s["plan"].h, s["level"], s["u1"], s["u2"], s["u"])
    else:
        E.eecmg_apply_H(s["plan"].handle, s["level"], s["x"], s["u"], s["transpose"])
    return s["u"]


def work(case):
    """Bytes: the data read and the result written once.  Flops: the convolutions (as 1-D passes
    where the PSF has factors) of the iterations that a restoration of noisy data takes at the
    least (r0, H r0, one H w per level) or that the case asks for, and the level start."""
    c = case
    if c["kind"] in ("batch", "serve"):
        parts = [work(d | {"kind": "restore"}) for d, _ in _items(c, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, dims = float(np.prod(_shape(c))), len(_shape(c))
    if c["psf"] in ("gauss", "gauss3"):
        conv = 2.0 * dims * (2 * c["band"] + 1)
    else:
        conv = 2.0 * float(np.count_nonzero(_psf(c)))
    start = {2: 250.0, 3: 700.0}[dims]
    kind = c["kind"].replace("vol_", "")
    if kind == "apply":
        return {"bytes": 8 * n, "flops": conv * n}
    if kind == "start":
        return {"bytes": 4 * n * (1 + 2.0 ** -dims + 4.0 ** -dims), "flops": start * n}
    if kind == "solve":
        return {"bytes": 12 * n, "flops": (2 + c["m"] * (2 if c.get("smoother") == "cgls" else 1)) * conv * n}
    return {"bytes": 8 * n, "flops": (3 * conv + start) * n / (1 - 2.0 ** -dims)}


# ------------------------------------------------------------------ the method in 64 bits


def _conv(x, k):
    """y(i) = sum_p K(p) x(i - p), zero outside: any dimension."""
    r = [s // 2 for s in k.shape]
    xp = torch.nn.functional.pad(x, [v for s in reversed(r) for v in (s, s)])
    y = torch.zeros_like(x)
    for at in np.argwhere(k != 0.0):
        y.add_(xp[tuple(slice(2 * s - int(p), 2 * s - int(p) + n) for s, p, n in zip(r, at, x.shape))], alpha=float(k[tuple(at)]))
    return y


def _flip(k):
    return np.ascontiguousarray(k[(slice(None, None, -1),) * k.ndim])


def _coarse(k, rho):
    return rho * k[tuple(slice((s // 2) % 2, None, 2) for s in k.shape)]


def _schedule(L):
    m = []
    for l in range(1, L + 1):
        t = (L - L / 2) ** 2 * 4.0 ** (L - l) if l > L / 2 else (L - 1.5 * l) * 4.0 ** (l - 1)
        m.append(max(1, math.ceil(t)))
    return m


def _solve(k, g, u, m, limit, smoother):
    """MR-II (three-term form) or CGLS from u: at most m iterations, none once ||r|| <= limit."""
    dot = lambda a, b: float((a * b).sum())  # noqa: E731
    r = g - _conv(u, k)
    limit = max(limit, 1e-5 * float(g.norm()))
    if m < 1 or float(r.norm()) <= limit:
        return u
    if smoother == "cgls":
        s = _conv(r, _flip(k))
        p, gamma = s, dot(s, s)
        for j in range(m):
            q = _conv(p, k)
            a = gamma / dot(q, q)
            u, r = u + a * p, r - a * q
            if j == m - 1 or float(r.norm()) <= limit:
                break
            s = _conv(r, _flip(k))
            new = dot(s, s)
            p, gamma = s + (new / gamma) * p, new
        return u
    p = _conv(r, k)
    q = _conv(p, k)
    p0 = q0 = None
    for j in range(m):
        if j:
            if float(r.norm()) <= limit:
                break
            z = _conv(q, k)
            b = dot(z, q) / dot(q, q)
            p1, q1 = q - b * p, z - b * q
            if q0 is not None:
                b = dot(z, q0) / dot(q0, q0)
                p1, q1 = p1 - b * p0, q1 - b * q0
            p0, q0, p, q = p, q, p1, q1
        a = dot(r, q) / dot(q, q)
        u, r = u + a * p, r - a * q
    return u


def _pi(u1, u2):
    """u1 plus a quarter of the multilinear interpolant of the coarser level's differences."""
    d = u1[(slice(None, None, 2),) * u1.dim()] - u2
    for ax, n in enumerate(u1.shape):
        i = torch.arange(n, device=d.device)
        a = i // 2
        b = torch.where(i % 2 == 1, (a + 1).clamp(max=d.shape[ax] - 1), a)
        d = 0.5 * (d.index_select(ax, a) + d.index_select(ax, b))
    return u1 + 0.25 * d


def _quadratic(ut, shape):
    q = torch.tensor([[1, 0, 0], [0.375, 0.75, -0.125], [0, 1, 0], [-0.125, 0.75, 0.375]], dtype=ut.dtype, device=ut.device)
    for ax, n in enumerate(shape):
        i = torch.arange(n, device=ut.device)
        wt = q[i % 4]
        got = 0
        for j in range(3):
            at = (2 * (i // 4) + j).clamp(max=ut.shape[ax] - 1)
            got = got + wt[:, j].reshape([-1 if a == ax else 1 for a in range(len(shape))]) * ut.index_select(ax, at)
        ut = got
    return ut


def _smooth(u):
    """The weighted plane fit over the in-image 3^n neighbourhood (raw moments, centred at the
    end; the moment matrix inverted on its eigenvalues above 1e-6 of the weight)."""
    n = u.dim()
    pad = torch.nn.functional.pad(u[None], [1, 1] * n)[0] if n < 4 else u
    ones = torch.nn.functional.pad(torch.ones_like(u)[None], [1, 1] * n)[0]
    W, vb = torch.zeros_like(u), torch.zeros_like(u)
    o, c = [torch.zeros_like(u) for _ in range(n)], [torch.zeros_like(u) for _ in range(n)]
    M = {(a, b): torch.zeros_like(u) for a in range(n) for b in range(a, n)}
    for at in np.ndindex(*(3,) * n):
        sl = tuple(slice(p, p + s) for p, s in zip(at, u.shape))
        v = pad[sl] - u
        wt = torch.exp(-(v * v)) * ones[sl]
        W += wt
        wv = wt * v
        vb += wv
        off = [p - 1 for p in at]
        for a in range(n):
            if off[a]:
                o[a].add_(wt, alpha=off[a])
                c[a].add_(wv, alpha=off[a])
                for b in range(a, n):
                    if off[b]:
                        M[a, b].add_(wt, alpha=off[a] * off[b])
    vb /= W
    for a in range(n):
        o[a] /= W
    for a in range(n):
        c[a] -= W * o[a] * vb
        for b in range(a, n):
            M[a, b] -= W * o[a] * o[b]
    thr = 1e-6 * W
    z = list(o)
    for _ in range(2 if n == 2 else 7):  # cyclic Jacobi rotations, applied to c and o
        for a in range(n):
            for b in range(a + 1, n):
                apq = M[a, b]
                zero = apq == 0
                th = (M[b, b] - M[a, a]) / (2 * torch.where(zero, torch.ones_like(apq), apq))
                t = torch.where(th >= 0, 1.0, -1.0) / (th.abs() + torch.sqrt(th * th + 1))
                t = torch.where(zero, torch.zeros_like(t), t)
                co = torch.rsqrt(t * t + 1)
                si = t * co
                M[a, a], M[b, b] = M[a, a] - t * apq, M[b, b] + t * apq
                M[a, b] = torch.zeros_like(apq)
                for r in range(n):
                    if r != a and r != b:
                        ka, kb = (min(r, a), max(r, a)), (min(r, b), max(r, b))
                        M[ka], M[kb] = co * M[ka] - si * M[kb], si * M[ka] + co * M[kb]
                c[a], c[b] = co * c[a] - si * c[b], si * c[a] + co * c[b]
                z[a], z[b] = co * z[a] - si * z[b], si * z[a] + co * z[b]
    out = u + vb
    for a in range(n):
        keep = M[a, a] > thr
        out -= torch.where(keep, c[a] * z[a] / torch.where(keep, M[a, a], torch.ones_like(out)), torch.zeros_like(out))
    return out


def _denoise(u):
    n = u.dim()
    grad2 = torch.zeros_like(u)
    for ax in range(n):
        lo, hi = u.narrow(ax, 0, 1), u.narrow(ax, u.shape[ax] - 1, 1)
        e = torch.cat([lo, u, hi], ax)
        grad2 += (0.5 * (e.narrow(ax, 2, u.shape[ax]) - e.narrow(ax, 0, u.shape[ax]))) ** 2
    c = 1.0 / (1.0 + grad2 / KPM ** 2)
    f = torch.zeros_like(u)
    for ax in range(n):
        if u.shape[ax] > 1:
            m = u.shape[ax] - 1
            flux = 0.5 * (c.narrow(ax, 0, m) + c.narrow(ax, 1, m)) * (u.narrow(ax, 1, m) - u.narrow(ax, 0, m))
            f.narrow(ax, 0, m).add_(flux)
            f.narrow(ax, 1, m).sub_(flux)
    return u + TAU * f


def _start(u1, u2, shape):
    return _denoise(_smooth(_quadratic(_pi(u1, u2), shape)))


def _cascade(g, psf, delta, L, smoother):
    gs, ks = [g], [psf]
    for _ in range(L - 1):
        fine = gs[0]
        gs.insert(0, fine[(slice(None, None, 2),) * g.dim()].contiguous())
        ks.insert(0, _coarse(ks[0], fine.numel() / gs[0].numel()))
    us = []
    for l, m in enumerate(_schedule(L)):
        u = torch.zeros_like(gs[l]) if l < 2 else _start(us[l - 1], us[l - 2], gs[l].shape)
        us.append(_solve(ks[l], gs[l], u, m, 1.1 * delta * math.sqrt(gs[l].numel()), smoother))
    return us[-1]


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("batch", "serve"):
        got = []
        for d, s in _items(c, seed):
            _, g, delta = _degraded(_shape(d), _psf(d), d["v"], s)
            got.append(_cascade(g.double(), _psf(d), delta, d["levels"], "mr2"))
        return got
    if kind in ("start", "vol_start"):
        u1, u2 = _start_inputs(c, seed)
        return _start(u1.double(), u2.double(), _shape(c))
    clean, g, delta = _degraded(_shape(c), _psf(c), c["v"], seed)
    if kind == "apply":
        return _conv(clean.double(), _flip(_psf(c)) if c["transpose"] else _psf(c))
    smoother = c.get("smoother", "mr2")
    if kind in ("solve", "vol_solve"):
        return _solve(_psf(c), g.double(), g.double(), c["m"], 0.0, smoother)
    return _cascade(g.double(), _psf(c), delta, c["levels"], smoother)
