"""The FP64 launches' dispatch and their edges against the oracle: three warps to 32 faces up to three face warps per
SM (84 x 85 on 152 SMs), one warp beyond (85 x 85); blocks of one to four warps; partly filled last warps of cells (8) and
faces (32);
every boundary kind; and the erfc / exp table from its first node to beyond its end (sqrt(lam) |U| = 6)."""
import numpy as np
import pytest

import oracle
from paper_1412_4489_gb300 import gks
from test_gpu_parity import BCSETS, _oracle_bc, _oracle_params, _perturbed, _rel_linf, _run_both, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bcname", list(BCSETS))
@pytest.mark.parametrize("shape", [(33, 3), (211, 23), (84, 85), (85, 85), (9, 641), (97, 90)])
def test_steps_match_the_oracle(shape, bcname):
    for mu, Pr in ((0.0, 1.0), (1e-3, 0.72)):
        p = _perturbed(*shape, seed=6, bc=BCSETS[bcname], mu=mu, Pr=Pr)
        g, o = _run_both(p, 2)
        for a, b in zip(g, o):
            assert _rel_linf(a, b) < 1e-11  # two steps of the 1e-12 that a step's faces are held to


@pytest.mark.parametrize("speed", [0.0, 1e-9, 0.03, 1.0, 5.0, 8.3, 8.6, 12.0, 40.0])
def test_half_space_moments_at_any_speed(speed):
    """sqrt(lam) |U| up to 28 (p / rho near 1): both sides of every face, both directions of flow."""
    for sign in (1.0, -1.0):
        p = _perturbed(13, 9, seed=8, amp=0.02)
        for a in (p.U, p.Wx, p.Wy):
            u = sign * speed - 1.0  # on top of the wave's velocity 1
            a[3] += u * a[1] + 0.5 * u * u * a[0]
            a[1] += u * a[0]
        dt = 0.2 * oracle.dt2d(_oracle_params(p), _state(p), 1.0)
        s = gks.Solver(p)
        got = gks.gks_debug_flux(s.h, p.nx, p.ny, dt)
        s.close()
        want = oracle.flux2d(_oracle_params(p), _state(p), _oracle_bc(p), dt)
        for a, b in zip(got, want):
            # both sides' rounding grows with the kinetic energy's share of the total
            assert np.max(np.abs(a - b)) <= 1e-12 * (1.0 + speed * speed) * np.max(np.abs(b))
