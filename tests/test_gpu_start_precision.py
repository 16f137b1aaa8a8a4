"""The level start's arithmetic where a faster approximation would show: the diffusivities'
quotient is correctly rounded, and weights below 2^-126 are kept."""
import numpy as np
import pytest

from gpu_helpers import dev, host, require_gpu

pytestmark = pytest.mark.gpu
F = np.float32


@pytest.fixture(scope="module")
def gpu():
    return require_gpu()


# A gradient of 1.5e19 squares to 2.3e38, within the range; twice it does not.
def test_volume_gradients_are_not_doubled_before_they_are_squared(gpu):
    torch, E = gpu
    b, k = 3e19, 100.0
    plan = E.VolumePlan(1, 1, 2, 1, np.ones((1, 1, 1)), 0.15, k)
    x, y = dev(torch, np.array([0.0, b])), torch.empty(2, device="cuda")
    E.eecmg_vol_denoise(plan.h, 0, x, y)
    g = np.float64(F(b)) / 2
    # a dozen roundings
    assert host(y)[0] == pytest.approx(0.15 * (k / g) ** 2 * 2 * g, rel=2.0 ** -20, abs=0)
    plan.close()
