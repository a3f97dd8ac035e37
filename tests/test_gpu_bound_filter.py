"""The CFL bound and the physical check of a state that goes in, where FP32 decides which cells need FP64: cells that
FP32 cannot judge (its range, its few bits there, near vacuum, bounds within its margin) among ordinary ones."""
import numpy as np
import pytest

from paper_1412_4489_gb300 import gks

pytestmark = pytest.mark.gpu

N = 1024  # 4,096 blocks: the last cells are loaded when the bound of the first ones is known


def _grid(cell, gamma, prec=gks.GKS_FP64):
    """A uniform flow with one other cell (rho, u, E) in the last row; (handle, cells)."""
    rho, u, E = np.ones((N, N)), np.full((N, N), 2.0), np.full((N, N), 20.0)
    rho[-1, -7], u[-1, -7], E[-1, -7] = cell
    U = np.stack([rho, rho * u, np.zeros((N, N)), E])
    h = gks.gks_create(N, N, 1.0, 1.0, gamma, 1.0, 0.0, options=gks.gks_default_options(prec))
    return h, U


def _bound(U, gamma):
    rho, m, _, E = U
    u = m / rho
    c = np.sqrt(gamma * (gamma - 1.0) * (E - 0.5 * m * u) / rho)
    return np.min(1.0 / ((np.abs(u) + c) * N))


@pytest.mark.parametrize("prec", [gks.GKS_FP64, gks.GKS_FP32_BULK])
@pytest.mark.parametrize("cell", [(1.0, 2.001, 20.003), (1.0, 2.0, 20.02), (1e-25, 50.0, 2e-22), (1e-12, 50.0, 1.3e-9),
                                  (1e25, 50.0, 2e28), (1.0, 50.0, 1250.001), (1e-20, 3.0, 1.0)])
def test_bound_of_every_cell(cell, prec):
    gamma = 1.4
    h, U = _grid(cell, gamma, prec)
    gks.gks_set_state(h, U)
    got = gks.gks_part_bound(h)
    back = np.zeros_like(U)
    gks.gks_get_state(h, back)
    gks.gks_destroy(h)
    # the state as it is held (FP32-bulk: pairs of FP32 numbers); E - kinetic energy cancels to 1e-6 at worst here
    assert got == pytest.approx(_bound(back, gamma), rel=1e-9)


@pytest.mark.parametrize("cell", [(2.0 ** 100, 1e20, 1e75), (1e100, 50.0, 2e103)])
def test_bound_beyond_fp32(cell):
    h, U = _grid(cell, 1.4)
    gks.gks_set_state(h, U)
    got = gks.gks_part_bound(h)
    gks.gks_destroy(h)
    assert got == pytest.approx(_bound(U, 1.4), rel=1e-9)


def _tiny():
    """p < 0, but 7 against 6 units of FP32's smallest number."""
    rho, kin = 1e-17, 6.7 * 2.0 ** -149
    return rho, np.sqrt(2.0 * kin / rho), 0.999 * kin


@pytest.mark.parametrize("cell", [_tiny(), (1.0, 2.0, 2.0 - 1e-9), (-1.0, 2.0, 20.0), (0.0, 0.0, 20.0),
                                  (float("nan"), 2.0, 20.0), (1.0, 2.0, float("inf")), (1e-30, 50.0, 1.2e-27)])
def test_a_state_that_is_not_physical_is_found(cell):
    h, U = _grid(cell, 2.9)
    with pytest.raises(gks.GKSError) as e:
        gks.gks_set_state(h, U)
    assert e.value.status == gks.GKS_ENONPHYSICAL
    gks.gks_destroy(h)
