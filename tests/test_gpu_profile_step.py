"""A profiled step: one name for each kernel, all of them timed, and the step that gks_step takes."""
import numpy as np
import pytest

from paper_1412_4489_gb300 import gks, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [gks.GKS_FP64, gks.GKS_FP32_BULK])
@pytest.mark.parametrize("mu", [0.0, 1e-3])
def test_names_and_state(prec, mu):
    p = wl.smooth_wave_2d(96, ny=70, seed=2)
    p.mu = mu
    a, b = gks.Solver(p, prec), gks.Solver(p, prec)
    for _ in range(3):
        ms = gks.gks_profile_step(a.h, 0.5)
        b.step(0.5)
        assert list(ms) == ["recon", "flux_x", "flux_y", "update", "finish"]
        assert all(0.0 < x < 1000.0 for x in ms.values())
    for x, y in zip(a.state()[:3], b.state()[:3]):
        assert np.array_equal(x, y)
    a.close()
    b.close()
