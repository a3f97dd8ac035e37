"""FP64 paths that small grids or ordinary data do not reach, against the oracle: the one-warp face launch over the range of
dt / tau; characteristic reconstruction of more block rows than a launch grid's y extent; the positivity check of the
reconstruction where FP32 cannot decide it."""
import numpy as np
import pytest

import oracle
from paper_1412_4489_gb300 import gks, workloads as wl
from test_gpu_face_regimes import CASES
from test_gpu_parity import _oracle_bc, _oracle_params, _perturbed, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mu,Pr,tau_eps", CASES)
def test_one_warp_faces_at_every_collision_time(mu, Pr, tau_eps):
    """97 x 90: beyond three face warps per SM, where three warps no longer share 32 faces."""
    dt = 1e-3
    p = _perturbed(97, 90, seed=5, mu=mu, Pr=Pr)
    P = oracle.params(gamma=p.gamma, mu=mu, Pr=Pr, tau_eps=tau_eps)
    want = oracle.flux2d(P, _state(p), _oracle_bc(p), dt)
    s = gks.Solver(p, tau_eps=tau_eps)
    got = gks.gks_debug_flux(s.h, p.nx, p.ny, dt)
    s.close()
    for a, b in zip(got, want):  # the bound of the small grid's test, whose derivation holds for any grid
        assert np.max(np.abs(a - b)) <= 1e-11 * np.max(np.abs(b))


@pytest.mark.parametrize("ny", [65535, 65536, 66000])
def test_characteristic_reconstruction_of_many_rows(ny):
    p = _perturbed(2, ny, seed=1)
    s = gks.Solver(p, characteristic=1)
    got = gks.gks_debug_recon(s.h, p.nx, p.ny)
    s.close()
    want = oracle.recon2d(_oracle_params(p, characteristic=1), _state(p), _oracle_bc(p))
    scale = np.abs(want).reshape(4, 6, -1).max(axis=2)[:, :, None, None] + 1e-300
    np.testing.assert_allclose(got / scale, want / scale, rtol=0, atol=1e-12)


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_positivity_check_where_fp32_cannot_tell(seed):
    """Pressures of 1e-8 to 1e-5 of the energy: far below what FP32 resolves of it, spread so widely that the polynomial's
    pressure is negative at one or more of the face centres of many cells; ordinary cells beside them."""
    n = 64
    rng = np.random.default_rng(seed)
    p = wl.smooth_wave_2d(n, seed=2)
    pres = 10.0 ** rng.uniform(-8.0, -5.0, (n, n))
    pres[:, n // 2:] = 1.0 + 0.1 * rng.uniform(-1, 1, (n, n // 2))
    pres[::7] = 1.0
    p.U[0], p.U[1], p.U[2] = 1.0, 1.0, 0.5
    p.U[3] = pres / (p.gamma - 1.0) + 0.625
    for a in (p.Wx, p.Wy):
        a[...] = np.array([1.0, 1.0, 0.5, 0.625 + 1e-6]).reshape(4, 1, 1, 1)
    s = gks.Solver(p)
    got = gks.gks_debug_recon(s.h, n, n)
    s.close()
    want = oracle.recon2d(_oracle_params(p), _state(p), _oracle_bc(p))
    dropped = np.all(want[:, 1:] == 0.0, axis=(0, 1))
    assert 50 < np.sum(dropped[:, :n // 2]) < n * n // 2 - 50
    assert np.array_equal(np.all(got[:, 1:] == 0.0, axis=(0, 1)), dropped)
    scale = np.abs(want).reshape(4, 6, -1).max(axis=2)[:, :, None, None] + 1e-300
    np.testing.assert_allclose(got / scale, want / scale, rtol=0, atol=1e-12)
