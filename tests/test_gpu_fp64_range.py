"""FP64 states whose density and pressure lie where rho^2 p under- or overflows FP64, against the oracle: in the split
face launch (up to three face warps per SM), the one-warp launch and the batched form."""
import numpy as np
import pytest

import oracle
from paper_1412_4489_gb300 import gks
from test_gpu_parity import _oracle_bc, _oracle_params, _perturbed, _rel_linf, _run_both, _state

pytestmark = pytest.mark.gpu


def _scaled(nx, ny, scale, mu=0.0, uniform=False):
    p = _perturbed(nx, ny, seed=6, mu=mu * scale, Pr=0.72 if mu else 1.0)
    for a in (p.U, p.Wx, p.Wy):
        if uniform:
            a[...] = np.array([1.0, 0.3, -0.2, 2.7]).reshape((4,) + (1,) * (a.ndim - 1))
        a *= scale
    return p


@pytest.mark.parametrize("shape", [(11, 7), (97, 90)])
@pytest.mark.parametrize("mu", [0.0, 1e-3])
@pytest.mark.parametrize("exponent", [-500, -400, -340, -250])
def test_small_states(shape, mu, exponent):
    p = _scaled(*shape, 2.0 ** exponent, mu)
    g, o = _run_both(p, 2)
    for a, b in zip(g, o):
        assert _rel_linf(a, b) < 1e-11  # two steps of the 1e-12 that a step's faces are held to


@pytest.mark.parametrize("shape", [(11, 7), (97, 90)])
@pytest.mark.parametrize("exponent", [250, 340, 400])
def test_large_uniform_states(shape, exponent):
    """Uniform: differences of such values have squares that overflow in the reconstruction's indicator."""
    p = _scaled(*shape, 2.0 ** exponent, uniform=True)
    g, o = _run_both(p, 2)
    for a, b in zip(g, o):
        assert _rel_linf(a, b) < 1e-11


def test_small_states_in_a_batch():
    p = _scaled(33, 18, 2.0 ** -400, 1e-3)
    b = gks.Batch([p])
    b.step(2, 0.5)
    b.sync()
    got = b.state(0)[:3]
    b.close()
    st = _state(p)
    for _ in range(2):
        assert oracle.step2d(_oracle_params(p), st, _oracle_bc(p), 0.5)[0] == 0
    for a, c in zip(got, (st.U, st.Wx, st.Wy)):
        assert _rel_linf(a, c) < 1e-11
