"""The device wait between the positivity fallback's passes: it runs out as a status and leaves the state and the handle
usable, and it never runs out because other handles' steps run beside it."""
import threading

import numpy as np
import pytest

from paper_1412_4489_gb300 import gks, workloads as wl

pytestmark = pytest.mark.gpu

QUADS = [(0.746, -0.312, 0.887, 0.312), (0.827, 0.438, -0.155, 0.861), (1.15, 0.953, 0.354, 0.494),
         (0.228, -0.698, -0.347, 1.304)]


def _problem(nx=16, ny=80):
    """Data on which the fallback fires (16 x 80: steps 3 and 5 in FP64)."""
    p = wl.riemann_2d(nx, ny, quadrants=QUADS, mu=9.4e-4, Pr=0.72)
    p.bc = [(wl.BC_PERIODIC, 0.0, 0.0, 1.0)] * 4
    return p


@pytest.mark.parametrize("prec", [gks.GKS_FP64, gks.GKS_FP32_BULK])
@pytest.mark.parametrize("block", [0, 3])
def test_a_wait_that_runs_out_fails_the_step_and_keeps_the_state(prec, block):
    """Block 0 also ends the step; block 3 is one of the others."""
    p = _problem()
    s, ref = gks.Solver(p, prec), gks.Solver(p, prec)
    gks.gks_set_wait_limit(s.h, 0.05, block)
    for taken in range(8):
        before = ref.state()
        try:
            s.step(0.5)
        except gks.GKSError as e:
            assert e.status == gks.GKS_ETIMEOUT and "wait" in gks.gks_last_error(s.h)
            break
        ref.step(0.5)
    else:
        pytest.fail("the fallback did not fire")
    assert 1 <= taken
    got = [np.zeros_like(a) for a in before[:3]]
    assert gks.load().gks_get_state(s.h, *(gks._ptr(a) for a in got), None) == gks.GKS_ETIMEOUT
    for a, b in zip(got, before):
        assert np.array_equal(a, b)
    # queued steps report it too, and take no step; a new state clears it
    gks.gks_advance(s.h, 5, 0.5)
    with pytest.raises(gks.GKSError) as e:
        gks.gks_sync(s.h)
    assert e.value.status == gks.GKS_ETIMEOUT
    gks.gks_set_wait_limit(s.h, 2.0)
    gks.gks_set_state(s.h, p.U, p.Wx, p.Wy)
    gks.gks_advance(s.h, 8, 0.5)
    assert gks.gks_sync(s.h)[1] == 8
    gks.gks_set_state(ref.h, p.U, p.Wx, p.Wy)
    for _ in range(8):
        ref.step(0.5)
    for a, b in zip(s.state()[:3], ref.state()[:3]):
        assert np.array_equal(a, b)
    s.close()
    ref.close()


def test_limits_out_of_range_are_refused():
    s = gks.Solver(_problem())
    for seconds in (0.0, -1.0, float("nan"), float("inf")):
        with pytest.raises(gks.GKSError) as e:
            gks.gks_set_wait_limit(s.h, seconds)
        assert e.value.status == gks.GKS_EINVAL
    s.close()


@pytest.mark.parametrize("prec", [gks.GKS_FP64, gks.GKS_FP32_BULK])
def test_fallbacks_of_several_handles_at_once(prec):
    """Eight handles on their own streams and threads, each with a fallback grid as large as the device."""
    p = _problem(160, 800)
    ref = gks.Solver(p, prec)
    ref.advance(12, 0.5)
    want = ref.state()
    ref.close()
    out = [None] * 8

    def run(k):
        s = gks.Solver(p, prec)
        if k % 2:
            for _ in range(12):
                s.step(0.5)
        else:
            s.advance(12, 0.5)
        out[k] = s.state()
        s.close()

    threads = [threading.Thread(target=run, args=(k,)) for k in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for o in out:
        assert o is not None
        for a, b in zip(o, want):
            assert np.array_equal(a, b)
