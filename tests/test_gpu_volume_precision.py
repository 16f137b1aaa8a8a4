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
