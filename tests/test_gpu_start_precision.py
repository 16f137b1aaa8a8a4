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


def fma(a, b, c):
    """a b + c rounded once: the sum is exact in 113 bits; in the 64 of other machines' long doubles
    a second rounding is possible but rare (about 2^-40 a case)."""
    L = np.longdouble
    return (L(a) * L(b) + L(c)).astype(F)


# The step's operations one by one, every result rounded to 32 bits and the quotient exactly: any other
# rounding of c moves some of these pixels by a last bit.
def test_denoise_is_bitwise_its_rounded_operations(gpu):
    torch, E = gpu
    h, w, tau, kpm = 300, 500, F(0.2), F(3.0)
    rng = np.random.default_rng(21)
    u = rng.uniform(-4, 4, (h, w)).astype(F)
    plan = E.Plan(w, h, 1, np.ones((3, 3)) / 9, 0.2, 3.0)
    y = torch.empty(h, w, device="cuda")
    E.eecmg_denoise(plan.handle, 0, dev(torch, u), y)
    p = np.pad(u, 1, mode="edge")
    gx, gy = F(0.5) * (p[1:-1, 2:] - p[1:-1, :-2]), F(0.5) * (p[2:, 1:-1] - p[:-2, 1:-1])
    ik2 = F(1.0) / (kpm * kpm)
    c = F(1.0) / fma(fma(gx, gx, gy * gy), np.full_like(u, ik2), np.ones_like(u))
    q = np.pad(c, 1, mode="edge")

    def flux(di, dj):  # zero across the image's edge
        cn, un = (a[1 + di:h + 1 + di, 1 + dj:w + 1 + dj] for a in (q, p))
        return (F(0.5) * (c + cn)) * (un - u)

    ref = fma(np.full_like(u, tau), ((flux(0, 1) + flux(0, -1)) + flux(-1, 0)) + flux(1, 0), u)
    assert np.array_equal(host(y).astype(F), ref)
    plan.close()


# Two voxels: one gradient, one flux, no other rounding than those written here.
def test_volume_denoise_is_bitwise_its_rounded_operations(gpu):
    torch, E = gpu
    tau, kpm = F(0.15), 3.0
    rng = np.random.default_rng(22)
    plan = E.VolumePlan(1, 1, 2, 1, np.ones((1, 1, 1)), 0.15, kpm)
    ik2, ht, half = F(1.0 / (kpm * kpm)), F(0.5) * tau, F(0.5)
    for _ in range(200):
        u = rng.uniform(-4, 4, (2, 1, 1)).astype(F)
        y = torch.empty(2, 1, 1, device="cuda")
        E.eecmg_vol_denoise(plan.h, 0, dev(torch, u), y)
        a, b = u[0, 0, 0], u[1, 0, 0]
        g = half * (b - a)  # the gradient at both voxels
        c = F(1.0) / fma(g * g, ik2, F(1.0))
        f = (c + c) * (b - a)
        assert host(y)[0, 0, 0] == fma(ht, f, a) and host(y)[1, 0, 0] == fma(ht, -f, b)
    plan.close()


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


# Gradients whose square leaves the range: c = 1/inf = 0 and nothing moves; and c below 2^-126 (22 bits or
# more of it left): the flux it carries, c within a last bit of those, is exact to 2^-20.
@pytest.mark.parametrize("b,k", [(1e25, 10.0), (3e19, 2.0 ** 0.5)])
def test_denoise_at_the_ends_of_the_range(gpu, b, k):
    torch, E = gpu
    plan, vol = E.Plan(2, 1, 1, np.ones((1, 1)), 0.2, k), E.VolumePlan(1, 1, 2, 1, np.ones((1, 1, 1)), 0.2, k)
    x, y = dev(torch, np.array([0.0, b])), torch.empty(2, device="cuda")
    g = np.float64(F(b)) / 2
    with np.errstate(over="ignore"):
        c = 1.0 / np.float64(F(F(g) * F(g)) * F(1.0 / k ** 2)) if b < 1e20 else 0.0
    assert c < 2.0 ** -126
    for denoise, h in ((E.eecmg_denoise, plan.handle), (E.eecmg_vol_denoise, vol.h)):
        denoise(h, 0, x, y)
        assert host(y)[0] == pytest.approx(0.2 * c * b, rel=2.0 ** -20, abs=0) and host(y)[1] == F(b)
    plan.close()
    vol.close()


# From a centre of 0 and one neighbour v of weight w = exp(-v^2) < 2^-126 the fit is w v: a subnormal number
# of 12 bits or more.  The tolerance: half a unit of those, twice, and v^2 <= 97 at a rounding of 2^-24 or two.
@pytest.mark.parametrize("v", [9.4, 9.6, 9.75])
def test_weights_below_the_normal_range_count(gpu, v):
    torch, E = gpu
    want = F(v) * np.exp(-np.float64(F(v)) ** 2)
    assert 2.0 ** -137 < want < 2.0 ** -122
    plan, vol = E.Plan(2, 1, 1, np.ones((1, 1))), E.VolumePlan(2, 1, 1, 1, np.ones((1, 1, 1)))
    x, y = dev(torch, np.array([0.0, v])), torch.empty(2, device="cuda")
    for smooth, h in ((E.eecmg_smooth, plan.handle), (E.eecmg_vol_smooth, vol.h)):
        smooth(h, 0, x, y)
        assert host(y)[0] == pytest.approx(want, rel=2.0 ** -11, abs=0)
    plan.close()
    vol.close()


# The largest scales: between equal neighbours the weight is 1 and a constant stays.
@pytest.mark.parametrize("scale", [1e38, 3e38, 3.402823e38])
def test_a_constant_stays_at_every_scale(gpu, scale):
    torch, E = gpu
    x = torch.full((5, 7, 9), 5.0, device="cuda")
    plan, vol = E.Plan(9, 35, 1, np.ones((1, 1)), s_scale=scale), E.VolumePlan(9, 7, 5, 1, np.ones((1, 1, 1)), s_scale=scale)
    for smooth, h in ((E.eecmg_smooth, plan.handle), (E.eecmg_vol_smooth, vol.h)):
        y = torch.empty_like(x)
        smooth(h, 0, x, y)
        assert torch.equal(x, y)
    plan.close()
    vol.close()
