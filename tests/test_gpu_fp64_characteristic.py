"""The FP64 characteristic reconstruction (cell-size units, projections by the eigenvectors' structure) at odd and
thin grids, with cells that are not square, for every boundary kind, alone and in a batch."""
import pytest

import oracle
from paper_1412_4489_gb300 import gks, workloads as wl
from test_gpu_fp32_layout import _smooth
from test_gpu_parity import BCSETS, _oracle_bc, _oracle_params, _rel_linf, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bcname", list(BCSETS))
@pytest.mark.parametrize("shape", [(1, 40), (31, 2), (33, 9), (130, 7)])
def test_two_steps_match_the_oracle(shape, bcname):
    bc = BCSETS[bcname]
    if shape[0] == 1 and (bc[0][0] if isinstance(bc[0], tuple) else bc[0]) != wl.BC_PERIODIC:
        pytest.skip("a single cell across needs periodic sides")
    p = _smooth(*shape, bc, mu=2e-3 if sum(shape) % 2 else 0.0)
    P, st, obc = _oracle_params(p, characteristic=1), _state(p), _oracle_bc(p)
    s = gks.Solver(p, characteristic=1)
    for _ in range(2):
        s.step(0.3)
        rc, _ = oracle.step2d(P, st, obc, 0.3)
        assert rc == 0
    got = [s.state()[:3]]
    s.close()
    if shape[0] > 1:  # a batch takes no single-column grids
        b = gks.Batch([p, p], characteristic=1)
        b.step(2, 0.3)
        b.sync()
        got.append(b.state(1)[:3])
        b.close()
    # 2^-53 times some 10^3 operations in two steps, times up to 10^3 by which the nonlinear weights amplify it
    for g in got:
        for a, w in zip(g, (st.U, st.Wx, st.Wy)):
            assert _rel_linf(a, w) < 1e-10
