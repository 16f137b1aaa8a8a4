"""Marched separable convolutions of volumes, voxel by voxel: both row forms (two rows a thread up to
radius 4, one beyond), rows on and off 16 bytes, ranges that cross tiles of ragged height."""
import numpy as np
import pytest

from gpu_helpers import dev, host, rel_l2, require_gpu

pytestmark = pytest.mark.gpu

ROWS = {1: 28, 2: 28, 3: 28, 4: 28, 5: 12, 6: 12}  # rows of the marched tile of radius r
DEPTH = {1: 53, 2: 101, 3: 118, 4: 160, 5: 101, 6: 120}
H = 87  # off 28 and 12


@pytest.fixture(scope="module")
def gpu():
    return require_gpu()


def marched(torch, d, h, w, r):
    """The level has at least 2 r slices per block (two blocks an SM), so that its blocks march."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return -(-w // 64) * -(-h // ROWS[r]) * d >= 4 * r * sms


def factors(r, seed):
    f = np.random.default_rng(seed).uniform(0.1, 1, (3, 2 * r + 1))
    f = f + f[:, ::-1]
    return f / f.sum(1, keepdims=True)


def passes(x, f):
    """The separable sum in 64 bits, zero outside."""
    y = x.astype(np.float64)
    for axis in range(3):
        r = f.shape[1] // 2
        p = np.pad(y, [(r, r) if a == axis else (0, 0) for a in range(3)])
        y = sum(f[axis][k] * np.take(p, range(k, k + x.shape[axis]), axis) for k in range(2 * r + 1))
    return y


@pytest.mark.parametrize("r", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("w,xo,yo", [(198, 0, 0), (200, 0, 0), (200, 1, 0), (200, 0, 1)])
def test_marched_apply(gpu, r, w, xo, yo):
    torch, E = gpu
    shape = (DEPTH[r], H, w)
    assert marched(torch, *shape, r)
    f = factors(r, 31)
    plan = E.VolumePlan(w, H, shape[0], 1, np.einsum("i,j,k->ijk", *f), delta=1.0)
    x = np.random.default_rng(32).uniform(0, 255, shape).astype(np.float32)
    n = x.size
    xb, yb = (torch.full((n + 4,), float("nan"), device="cuda") for _ in range(2))
    xb[xo:xo + n] = dev(torch, x.reshape(-1))
    E.eecmg_vol_apply_H(plan.h, 0, xb[xo:xo + n], yb[yo:yo + n])
    # the taps' and three passes' roundings: 3 (2 r + 1) products and sums of at most 255
    got = host(yb)
    assert np.abs(got[yo:yo + n].reshape(shape) - passes(x, f)).max() <= 255 * (6 * r + 9) * 2.0 ** -24
    assert np.isnan(got[:yo]).all() and np.isnan(got[yo + n:]).all()
    plan.close()


@pytest.mark.parametrize("r,w", [(2, 198), (2, 200), (5, 198), (5, 200)])
def test_marched_solve_matches_oracle(gpu, orc, r, w):
    from paper_2311_03010_gb300 import synth

    torch, E = gpu
    d = DEPTH[r]
    assert marched(torch, d, H, w, r)
    psf = synth.gaussian_psf3(0.4 * r, r)
    p = synth.make_volume_problem(d, H, w, 33, psf, 0.01)
    plan = E.VolumePlan(w, H, d, 1, psf, stop="fixed")
    u = dev(torch, p.g)
    E.eecmg_vol_level_solve(plan.h, 0, dev(torch, p.g), u, 3)
    it, res = plan.stats()
    ref, k, rres = orc.mr2_3(psf, p.g.astype(np.float64), p.g.astype(np.float64), 3, 0.0, 1e-5)
    # the bars of the solves on other shapes
    assert it[0] == k == 3 and rel_l2(host(u), ref) <= 1e-4 and abs(res[0] - rres) <= 1e-4 * max(rres, 1.0)
    plan.close()
