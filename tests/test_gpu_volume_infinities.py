"""A PSF applied by whole rows of taps: an infinite or NaN voxel reaches the outputs that a tap of
weight other than zero carries it to, and no others."""
import numpy as np
import pytest

from gpu_helpers import dev, host, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    return require_gpu()


# a 7-point star and a band: rows of taps with zeros at their ends; widths off and on 4, the voxel inside
# and at a corner
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("shape,at", [((9, 14, 66), (4, 6, 30)), ((9, 14, 68), (0, 0, 0)), ((40, 20, 130), (39, 19, 129))])
@pytest.mark.parametrize("r", [1, 2])
def test_non_finite_voxels_stay_within_the_taps(gpu, r, shape, at, bad):
    torch, E = gpu
    k = np.zeros((2 * r + 1,) * 3)
    for axis in range(3):
        i = [r, r, r]
        for i[axis] in range(2 * r + 1):
            k[tuple(i)] = 1.0 + (i[axis] == r)
    k /= k.sum()
    x = np.random.default_rng(51).uniform(1, 2, shape).astype(np.float32)
    x[at] = bad
    plan = E.VolumePlan(shape[2], shape[1], shape[0], 1, k, delta=1.0)
    y = torch.empty(shape, device="cuda")
    E.eecmg_vol_apply_H(plan.h, 0, dev(torch, x), y)
    ref = np.zeros(shape)
    p = np.pad(x.astype(np.float64), r)
    for i in np.argwhere(k != 0):
        ref += k[tuple(i)] * p[tuple(slice(a, a + n) for a, n in zip(i, shape))]
    assert np.allclose(host(y), ref, rtol=(np.count_nonzero(k) + 2) * 2.0 ** -24, atol=0, equal_nan=True)
    plan.close()
