"""The face evolution over the range of dt / tau that its branches split: exp(-dt/tau) exactly zero (and
its exponential skipped in FP64), the closed forms of the time weights, their series, on both sides of the
line between the two, for Euler and Navier-Stokes faces with and without the Prandtl correction."""
import numpy as np
import pytest

import oracle
from paper_1412_4489_gb300 import gks, workloads as wl

pytestmark = pytest.mark.gpu


def _problem(mu, Pr, gamma):
    """A periodic wave with a jump in pressure and tangential velocity in every row."""
    p = wl.smooth_wave_2d(11, ny=7, seed=4, gamma=gamma)
    rng = np.random.default_rng(7)
    for a in (p.U, p.Wx, p.Wy):
        a[2] += 0.1 * a[0]
        a[3] += 0.1 * a[1] + 0.005 * a[0]
        a *= 1.0 + 0.01 * rng.uniform(-1.0, 1.0, a.shape)
    p.mu, p.Pr = mu, Pr
    return p


# dt / tau with p near 1: Euler tau_eps dt, Navier-Stokes mu / p, plus the pressure jump's share (about 0.01 dt)
CASES = [(0.0, 1.0, 0.0), (0.0, 1.0, 0.0005), (0.0, 0.72, 0.02), (0.0, 1.0, 0.45), (0.0, 1.0, 0.6), (0.0, 0.72, 1.9),
         (0.0, 1.0, 2.2), (0.0, 1.0, 8.0), (1e-6, 1.0, 0.0), (1e-4, 0.72, 0.0), (1.8e-3, 0.72, 0.0), (2.1e-3, 1.0, 0.0),
         (5e-3, 0.72, 0.0), (1e-2, 1.0, 0.0)]


@pytest.mark.parametrize("gamma", [1.4, 5.0 / 3.0])
@pytest.mark.parametrize("mu,Pr,tau_eps", CASES)
def test_face_evolution_at_every_collision_time(mu, Pr, tau_eps, gamma):
    dt = 1e-3
    p = _problem(mu, Pr, gamma)
    P = oracle.params(gamma=gamma, mu=mu, Pr=Pr, tau_eps=tau_eps)
    st = oracle.State2D(p.nx, p.ny, p.Lx, p.Ly, p.U, p.Wx, p.Wy)
    want = oracle.flux2d(P, st, oracle.bcs([b[0] for b in p.bc], [b[1:] for b in p.bc]), dt)
    # the oracle's closed forms lose (tau / dt)^3 roundings at long collision times (at most 10^3 here); the
    # FP32 form rounds every operand: 2^-24 times some tens of operations on values of order 1..10
    for prec, tol in ((gks.GKS_FP64, 1e-11), (gks.GKS_FP32_BULK, 1e-5)):
        s = gks.Solver(p, prec, tau_eps=tau_eps)
        got = gks.gks_debug_flux(s.h, p.nx, p.ny, dt)
        s.close()
        for a, b in zip(got, want):
            assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b))
