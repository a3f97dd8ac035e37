"""The rounding errors that FP32 steps add up to on a smooth wave (both face directions, many steps), against FP64."""
import numpy as np
import pytest

from paper_1412_4489_gb300 import gks, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,steps", [(701, 499, 48), (128, 96, 96)])
def test_rounding_errors_add_up_no_faster_than_in_the_batched_form(nx, ny, steps):
    """The batched form takes the same steps with moments in the fixed frame.  The single grid's routine rounds each
    face less, so its accumulated error may not be the larger one; a tenth is left for the draw of the phase."""
    p = wl.smooth_wave_2d(nx, ny=ny, seed=2)
    runs = []
    for prec in (gks.GKS_FP64, gks.GKS_FP32_BULK):
        s = gks.Solver(p, prec, tau_eps=0.0)
        s.advance(steps, 0.5)
        runs.append(s.state()[:3])
        s.close()
    b = gks.Batch([p], gks.GKS_FP32_BULK, tau_eps=0.0)
    b.step(steps, 0.5)
    b.sync()
    runs.append(b.state(0)[:3])
    b.close()
    for want, single, batch in zip(*runs):
        assert np.linalg.norm(single - want) <= 1.1 * np.linalg.norm(batch - want)


def test_long_runs_keep_below_the_batched_form():
    """3,000 steps at the paper's CFL number: errors that repeat as the wave passes add up."""
    p = wl.smooth_wave_2d(512, seed=2)
    runs = []
    for prec in (gks.GKS_FP64, gks.GKS_FP32_BULK):
        s = gks.Solver(p, prec, tau_eps=0.0)
        s.advance(3000, 0.2)
        runs.append(s.state()[0])
        s.close()
    b = gks.Batch([p], gks.GKS_FP32_BULK, tau_eps=0.0)
    b.step(3000, 0.2)
    b.sync()
    runs.append(b.state(0)[0])
    b.close()
    want, single, batch = runs
    assert np.linalg.norm(single - want) <= 1.1 * np.linalg.norm(batch - want)
