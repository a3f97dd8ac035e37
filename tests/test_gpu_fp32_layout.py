"""The FP32 form's vector layout and its bulk-stored reconstruction records at their edges: rows shorter than, equal
to and past whole warps of cells, single rows and columns, every boundary kind (ghost records), both
reconstructions, and the state's way in and out."""
import numpy as np
import pytest

import oracle
from paper_1412_4489_gb300 import gks, workloads as wl
from test_gpu_parity import BCSETS, _oracle_bc, _oracle_params, _rel_linf, _state

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (1, 40), (31, 1), (32, 2), (33, 9), (63, 8), (64, 17), (97, 5), (130, 33)]


def _smooth(nx, ny, bc, mu):
    """A smooth wave in all four variables."""
    p = wl.smooth_wave_2d(nx, ny=ny, seed=9)
    for a in (p.U, p.Wx, p.Wy):
        rho = a[0].copy()
        v = 0.1 * (rho - 1.0)
        a[3] += 0.5 * rho * ((1.0 + v) ** 2 - 1.0) + 0.2 * (rho - 1.0)
        a[2] += rho * v
    p.bc = [b if isinstance(b, tuple) else (b, 0.0, 0.0, 1.0) for b in bc]
    p.mu, p.Pr = mu, 0.72 if mu else 1.0
    return p


@pytest.mark.parametrize("characteristic", [0, 1])
@pytest.mark.parametrize("bcname", list(BCSETS))
@pytest.mark.parametrize("shape", SHAPES)
def test_two_steps_match_the_oracle(shape, bcname, characteristic):
    nx, ny = shape
    bc = BCSETS[bcname]
    kinds = [b[0] if isinstance(b, tuple) else b for b in bc]
    if (nx == 1 and kinds[0] != wl.BC_PERIODIC) or (ny == 1 and kinds[2] != wl.BC_PERIODIC):
        pytest.skip("a single cell across needs periodic sides")
    p = _smooth(nx, ny, bc, mu=2e-3 if (nx + ny) % 2 else 0.0)
    P, st, obc = _oracle_params(p, characteristic=characteristic), _state(p), _oracle_bc(p)
    s = gks.Solver(p, gks.GKS_FP32_BULK, characteristic=characteristic)
    got = s.state()[:3]
    assert np.array_equal(got[0].astype(np.float32), p.U.astype(np.float32))
    assert np.array_equal(got[1], p.Wx.astype(np.float32)) and np.array_equal(got[2], p.Wy.astype(np.float32))
    for _ in range(2):
        s.step(0.3)
        rc, _ = oracle.step2d(P, st, obc, 0.3)
        assert rc == 0
    got = s.state()[:3]
    s.close()
    # 2^-24 of every operand and of some tens of operations a step, on values of order 1 to 10
    for a, b in zip(got, (st.U, st.Wx, st.Wy)):
        assert _rel_linf(a, b) < 2e-5
