"""What the volume solver holds in 64 bits and what its sums keep, on inputs whose exact
values a 32-bit or a double-float form cannot represent."""
import numpy as np
import pytest

from gpu_helpers import dev, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    return require_gpu()


# A zero start has r = g, so ||r||^2 = ||g||^2 exactly; a tolerance 2^-52 below 1 puts the limit 2^-51 below
# that, which 53 bits tell apart: one iteration.  Rounded to 48 bits the two are equal, and none runs.
@pytest.mark.parametrize("seed", range(8))
def test_the_stop_limit_has_53_bits(gpu, seed):
    torch, E = gpu
    rng = np.random.default_rng(seed)
    shape = (5, 9, 13)
    plan = E.VolumePlan(shape[2], shape[1], shape[0], 1, np.ones((1, 1, 1)), iters=[1], stop="fixed", conv_tol=1.0 - 2.0 ** -52)
    g = dev(torch, rng.uniform(1, 255, shape))
    plan.restore(g, torch.empty_like(g))
    assert plan.stats()[0] == [1]
    plan.close()


# Rows of 4096, 1, 1, 1 from u = 0: r = g exactly, and an FP32 sum of four squares drops the ones
# (2^24 + 1 rounds to 2^24): 1.8e-7 of ||r||^2.  One product at a time a compensated sum of n terms is
# off by n 2^-48 of it, 300 terms a thread here: 1.1e-12.  Marched (separable), dense and sparse PSFs.
@pytest.mark.parametrize("name", ["marched", "tiles", "dense", "sparse"])
@pytest.mark.parametrize("w", [256, 254])
def test_inner_products_keep_every_product(gpu, name, w):
    torch, E = gpu
    shape = (20, 30, w) if name == "tiles" else (160, 112, w)
    if name in ("marched", "tiles"):
        k = np.ones((3, 3, 3))
    elif name == "dense":
        k = np.ones((3, 3, 3))
        k[0, 0, 0] = k[2, 2, 2] = 2.0
    else:
        k = np.zeros((9, 9, 9))
        for i in range(9):
            k[i, i, i] = 1.0
    plan = E.VolumePlan(w, shape[1], shape[0], 1, k / k.sum(), stop="fixed")
    row = np.ones(w, np.float32)
    row[::4] = 4096.0
    g = np.broadcast_to(row, shape)
    u = torch.zeros(shape, device="cuda")
    E.eecmg_vol_level_solve(plan.h, 0, dev(torch, g), u, 0)
    rms = plan.stats()[1][0]
    assert rms == pytest.approx(np.sqrt(np.mean(row.astype(np.float64) ** 2)), rel=1e-11)
    plan.close()
