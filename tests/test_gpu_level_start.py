"""The strip kernel of the fused level start against the operator kernels it
fuses, at the widths and heights where its strips and segments end."""
import numpy as np
import pytest

from gpu_helpers import dev, host, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    return require_gpu()


# strips yield 116 columns and are interior from width 241 on; cells are 4 columns
@pytest.mark.parametrize("shape", [(1, 1), (2, 3), (9, 116), (9, 117), (6, 119), (13, 232), (13, 233), (40, 240),
                                   (40, 241), (41, 242), (37, 243), (1021, 1903), (2050, 1160)])
@pytest.mark.parametrize("scale", [1.0, 0.0])
def test_strips_equal_the_operator_chain(gpu, shape, scale):
    torch, E = gpu
    from paper_2311_03010_gb300 import synth

    h, w = shape
    plan = E.Plan(w, h, 3, synth.gaussian_psf(1.0, 2), s_scale=scale)
    h1, w1 = (h + 1) // 2, (w + 1) // 2
    rng = np.random.default_rng(7)
    u1 = (synth.synthetic_image(h1, w1, 58) + rng.normal(0, 1.5, (h1, w1))).astype(np.float32)
    u2 = (u1[::2, ::2] + rng.uniform(-3, 3, ((h1 + 1) // 2, (w1 + 1) // 2))).astype(np.float32)
    d1, d2 = dev(torch, u1), dev(torch, u2)
    # the outputs start one float into a buffer too: rows that are not 16-byte aligned
    fused = [torch.full((h * w + 4,), float("nan"), device="cuda") for _ in range(2)]
    views = [fused[0][:h * w], fused[1][1:h * w + 1]]
    for v in views:
        E.eecmg_start_level(plan.handle, 2, d1, d2, v)
    p, s, d = (torch.empty(h, w, device="cuda") for _ in range(3))
    E.eecmg_prolong(plan.handle, 2, d1, d2, p)
    E.eecmg_smooth(plan.handle, 2, p, s)
    E.eecmg_denoise(plan.handle, 2, s, d)
    for v in views:
        assert np.array_equal(host(v).reshape(h, w), host(d))
    for f, lo, hi in ((fused[0], 0, h * w), (fused[1], 1, h * w + 1)):  # nothing written past the level
        f = host(f)
        assert np.isnan(f[:lo]).all() and np.isnan(f[hi:]).all()
    plan.close()
