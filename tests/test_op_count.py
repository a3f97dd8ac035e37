"""The operation count of one face (host only): each precision's own arithmetic as the kernels run it."""
import numpy as np
import pytest

from paper_1412_4489_gb300 import gks


def _face(seed=1):
    rng = np.random.default_rng(seed)

    def cons():
        r, u, v, p = 1 + 0.1 * rng.uniform(), 0.3, -0.2, 1 + 0.1 * rng.uniform()
        return np.array([r, r * u, r * v, p / 0.4 + 0.5 * r * (u * u + v * v)])

    L, R = np.zeros((6, 4)), np.zeros((6, 4))
    L[0], R[0] = cons(), cons()
    L[1:], R[1:] = rng.normal(size=(2, 5, 4))
    return L, R, np.array([[cons() for _ in range(3)] for _ in range(2)])


def _count(prec, mu=0.0, Pr=1.0, tau_eps=0.05):
    return gks.gks_face_op_count(*_face(), 0.01, 0.01, 1e-3, 1.4, mu, Pr, tau_eps, 1.0, prec)


@pytest.mark.parametrize("mu,Pr", [(0.0, 1.0), (1e-3, 0.72)])
def test_quotients_and_special_functions(mu, Pr):
    """Both: 1 / rho0, the pressure jump's, dt / tau, and mu / p0 with viscosity; one root a side and exp(-dt/tau).
    FP64: one reciprocal and no library erfc or exp a side.  FP32: 1 / rho, rho / p, an erfc and an exp a side, and
    2 lam = 1 / s again in each of its two kinetic parts; at dt / tau = 1, the viscous case's, its time weights are series."""
    d, f = _count(gks.GKS_FP64, mu, Pr), _count(gks.GKS_FP32_BULK, mu, Pr)
    common = 3 + (mu > 0)
    assert (d["div"], d["erfc"], d["exp"], d["rsqrt"]) == (common + 2, 0, 1, 2)
    assert (f["div"], f["erfc"], f["exp"], f["rsqrt"]) == (common + 8, 2, 3 if mu == 0.0 else 2, 2)


def test_the_table_s_polynomials_are_counted():
    """22 additions and 20 multiplications a side, and the few operations around quotients."""
    d, f = _count(gks.GKS_FP64), _count(gks.GKS_FP32_BULK)
    assert 2 * 20 <= d["mul"] - f["mul"] <= 2 * 30
    assert 2 * 22 <= d["add"] - f["add"] <= 2 * 26
