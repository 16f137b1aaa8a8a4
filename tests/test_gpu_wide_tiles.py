"""Large convolution tiles: every pixel, inputs and outputs on and off 16 bytes."""
import numpy as np
import pytest

from gpu_helpers import dev, host, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    return require_gpu()


@pytest.mark.parametrize("band", [0, 1, 4, 5, 10, 12])
@pytest.mark.parametrize("h,w", [(16 * 56 + 1, 18 * 120 + 4), (900, 2276), (304 * 56 - 3, 12)])
def test_every_pixel_of_large_tiles(gpu, h, w, band):
    torch, E = gpu
    assert w % 4 == 0 and -(-h // 56) * -(-w // 120) >= 304  # large tiles
    rng = np.random.default_rng(41)
    f = rng.uniform(0.1, 1, (2, 2 * band + 1))
    f /= f.sum(1, keepdims=True)
    plan = E.Plan(w, h, 1, np.outer(*f), smoother="cgls", delta=1.0)
    x = rng.uniform(0, 255, (h, w)).astype(np.float32)
    pad = np.pad(x.astype(np.float64), ((band, band), (0, 0)))
    ref = sum(f[0][d] * pad[d:d + h] for d in range(2 * band + 1))
    pad = np.pad(ref, ((0, 0), (band, band)))
    ref = sum(f[1][d] * pad[:, d:d + w] for d in range(2 * band + 1))
    n = x.size
    for xo, yo in ((0, 0), (1, 0), (0, 1), (3, 2)):
        xb, yb = (torch.full((n + 4,), float("nan"), device="cuda") for _ in range(2))
        xb[xo:xo + n] = dev(torch, x.reshape(-1))
        E.eecmg_apply_H(plan.handle, 0, xb[xo:xo + n], yb[yo:yo + n], 1)
        got = host(yb)
        # the taps' and two passes' roundings: 2 (2 r + 1) products and sums of at most 255
        assert np.abs(got[yo:yo + n].reshape(h, w) - ref).max() <= 255 * (4 * band + 8) * 2.0 ** -24
        assert np.isnan(got[:yo]).all() and np.isnan(got[yo + n:]).all()
    plan.close()
