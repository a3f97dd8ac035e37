"""The FP32 batch's face routine (its own: moments in the fixed frame) against the oracle: over the range of dt / tau that
its branches split, Euler, Navier-Stokes, and both in one batch; every boundary kind; both reconstructions."""
import numpy as np
import pytest

import oracle
from paper_1412_4489_gb300 import gks, workloads as wl
from test_gpu_face_regimes import CASES, _problem
from test_gpu_fp32_layout import _smooth
from test_gpu_parity import BCSETS, _oracle_bc, _oracle_params, _rel_linf, _state

pytestmark = pytest.mark.gpu


def _stepped(ps, steps, cfl, **opts):
    b = gks.Batch(ps, gks.GKS_FP32_BULK, **opts)
    b.step(steps, cfl)
    b.sync()
    out = b.state(0)[:3]
    b.close()
    return out


@pytest.mark.parametrize("gamma", [1.4, 5.0 / 3.0])
@pytest.mark.parametrize("mu,Pr,tau_eps", CASES)
def test_one_step_at_every_collision_time(mu, Pr, tau_eps, gamma):
    dt = 1e-3
    p = _problem(mu, Pr, gamma)
    P, bc = oracle.params(gamma=gamma, mu=mu, Pr=Pr, tau_eps=tau_eps), _oracle_bc(p)
    cfl = dt / oracle.dt2d(P, _state(p), 1.0)
    Fx, Fy = oracle.flux2d(P, _state(p), bc, dt)[:2]
    st = _state(p)
    assert oracle.step2d(P, st, bc, cfl)[0] == 0
    other = wl.smooth_wave_2d(16, seed=2, gamma=gamma)
    other.mu, other.Pr = (0.0, 1.0) if mu else (1e-3, 0.72)
    dx, dy = p.Lx / p.nx, p.Ly / p.ny
    for ps in ([p], [p, other]):  # one model for all grids; decided grid by grid
        U, Wx, Wy = _stepped(ps, 1, cfl, tau_eps=tau_eps)
        # 1e-5 of each face's flux and point values, as the single grid's: 2^-24 times some tens of operations on values of
        # order 1 to 10; a cell's change sums its four faces' fluxes
        for v in range(4):
            tol = 1e-5 * 2.0 * (np.max(np.abs(Fx)) / dx + np.max(np.abs(Fy)) / dy)
            assert np.max(np.abs(U[v] - st.U[v])) <= tol
        for a, b in ((Wx, st.Wx), (Wy, st.Wy)):
            assert np.max(np.abs(a - b)) <= 1e-5 * np.max(np.abs(b))


@pytest.mark.parametrize("characteristic", [0, 1])
@pytest.mark.parametrize("bcname", list(BCSETS))
@pytest.mark.parametrize("shape", [(2, 40), (33, 9), (64, 17)])
def test_two_steps_with_every_boundary(shape, bcname, characteristic):
    for mu in (0.0, 2e-3):
        p = _smooth(*shape, BCSETS[bcname], mu)
        st = _state(p)
        for _ in range(2):
            assert oracle.step2d(_oracle_params(p, characteristic=characteristic), st, _oracle_bc(p), 0.3)[0] == 0
        # the single grid's bound for two such steps
        for a, b in zip(_stepped([p], 2, 0.3, characteristic=characteristic), (st.U, st.Wx, st.Wy)):
            assert _rel_linf(a, b) < 2e-5
