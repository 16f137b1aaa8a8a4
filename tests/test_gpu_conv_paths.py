"""The convolution paths that a size or a PSF's shape selects: large tiles, vertical
runs of taps, dense and sparse volume PSFs, against 64-bit sums of the same taps."""
import numpy as np
import pytest

from gpu_helpers import dev, host, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    return require_gpu()


def correlate(x, taps):
    """sum over (offset, weight) of weight x(i + offset), zero outside."""
    y = np.zeros(x.shape)
    for off, wt in taps:
        if any(abs(o) >= n for o, n in zip(off, x.shape)):
            continue
        src = tuple(slice(max(o, 0), n + min(o, 0)) for o, n in zip(off, x.shape))
        dst = tuple(slice(max(-o, 0), n + min(-o, 0)) for o, n in zip(off, x.shape))
        y[dst] += wt * x[src]
    return y


# FP32: (taps + 1) roundings of sums of at most 255 sum|K|; two passes round twice
def bar(k):
    return 255.0 * np.abs(k).sum() * (np.count_nonzero(k) + 2 * max(k.shape) + 4) * 2.0 ** -24


# From 304 tiles of 56 x 120 on, rows of whole float4s: exact fit, one row and quad over, one tile short, ragged
@pytest.mark.parametrize("h,w", [(16 * 56, 19 * 120), (16 * 56 + 1, 18 * 120 + 4), (304 * 56, 12), (303 * 56, 60), (900, 2278)])
@pytest.mark.parametrize("band", [0, 1, 4, 5, 10, 12])
def test_large_tiles(gpu, h, w, band):
    torch, E = gpu
    rng = np.random.default_rng(3)
    a, b = rng.uniform(0.1, 1, 2 * band + 1), rng.uniform(0.1, 1, 2 * band + 1)
    k = np.outer(a, b)
    k /= k.sum()
    x = rng.uniform(0, 255, (h, w)).astype(np.float32)
    plan = E.Plan(w, h, 1, k, smoother="cgls", delta=1.0)
    buf = torch.full((h * w + 4,), float("nan"), device="cuda")
    xd = dev(torch, x)
    for view in (buf[:h * w], buf[1:h * w + 1]):  # 16-byte aligned and not
        buf.fill_(float("nan"))
        E.eecmg_apply_H(plan.handle, 0, xd, view, 1)
        got = host(view).reshape(h, w)
        at = [0, 1, 55, 56, 57, h // 2, h - 2, h - 1]
        pad = np.pad(x.astype(np.float64), band)
        for i in [i for i in at if i < h]:  # whole rows, by 64-bit sums
            rows = sum(a[d] * pad[i + d] for d in range(2 * band + 1))
            ref = sum(b[d] * rows[d:d + w] for d in range(2 * band + 1)) / (a.sum() * b.sum())
            assert np.abs(got[i] - ref).max() <= bar(k), i
        assert np.isfinite(got).all() and int(torch.isnan(buf).sum()) == 4
    plan.close()


# vertical runs of 1, 2, 3, 4 and more taps, gaps inside a column, one tap
@pytest.mark.parametrize("name", ["line", "column9", "column5gap", "checker", "single"])
@pytest.mark.parametrize("shape", [(64, 64), (33, 70), (9, 130)])
def test_runs_of_taps(gpu, name, shape):
    torch, E = gpu
    rng = np.random.default_rng(4)
    k = np.zeros((9, 7))
    if name == "line":
        for i in range(7):
            k[1 + i:3 + i, i] = rng.uniform(0.1, 1, 2)
    elif name == "column9":
        k[:, 3] = rng.uniform(0.1, 1, 9)
        k[2:5, 5] = 0.3
    elif name == "column5gap":
        k[:, 1] = rng.uniform(0.1, 1, 9)
        k[4, 1] = 0.0
        k[0, 6] = 0.2
    elif name == "checker":
        k[::2, ::2] = rng.uniform(0.1, 1, (5, 4))
    else:
        k[2, 6] = 1.0
        k[7, 0] = 0.5
    k /= k.sum()
    h, w = shape
    x = rng.uniform(0, 255, (h, w)).astype(np.float32)
    plan = E.Plan(w, h, 1, k, smoother="cgls", delta=1.0)
    y = torch.empty(h, w, device="cuda")
    for tr in (0, 1):
        E.eecmg_apply_H(plan.handle, 0, dev(torch, x), y, tr)
        taps = [((p - 4) * (1 if tr else -1), (q - 3) * (1 if tr else -1)) for p, q in np.argwhere(k != 0)]
        ref = correlate(x.astype(np.float64), [(o, k[p, q]) for o, (p, q) in zip(taps, np.argwhere(k != 0))])
        assert np.abs(host(y) - ref).max() <= bar(k)
    plan.close()


# dense rows of taps, a sparse line in a large support, separable; widths off and on 4, slices fewer than the radius
@pytest.mark.parametrize("name", ["dense", "sparse", "sep"])
@pytest.mark.parametrize("shape", [(3, 5, 4), (20, 30, 64), (9, 33, 70), (2, 29, 131), (40, 17, 68)])
@pytest.mark.parametrize("r", [1, 2, 4, 6])
def test_volume_forms(gpu, name, shape, r):
    torch, E = gpu
    rng = np.random.default_rng(5)
    n = 2 * r + 1
    if name == "sep":
        f = [rng.uniform(0.1, 1, n) for _ in range(3)]
        f = [v + v[::-1] for v in f]
        k = f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]
    else:
        k = rng.uniform(0.1, 1, (n, n, n)) if name == "dense" else np.zeros((n, n, n))
        if name == "sparse":
            for i in range(n):
                k[i, i, i] = 1.0 + i
                k[i, n - 1 - i, r] += 0.5
        k = k + k[::-1, ::-1, ::-1]
    k /= k.sum()
    d, h, w = shape
    plan = E.VolumePlan(w, h, d, 1, k, delta=1.0)
    x = rng.uniform(0, 255, shape).astype(np.float32)
    y = torch.full(shape, float("nan"), device="cuda")
    E.eecmg_vol_apply_H(plan.h, 0, dev(torch, x), y)
    ref = correlate(x.astype(np.float64), [(tuple(int(v) - r for v in i), k[tuple(i)]) for i in np.argwhere(k != 0)])
    assert np.abs(host(y) - ref).max() <= bar(k)
    plan.close()
