"""Host arrays at any address: page-locked ones are read and written in place only where a kernel's 8-byte accesses may go."""
import numpy as np
import pytest

from paper_1412_4489_gb300 import gks, workloads as wl

pytestmark = pytest.mark.gpu


def _at(a, offset, pinned):
    """A copy of a that starts `offset` bytes past a multiple of 64."""
    import torch
    raw = torch.empty(a.nbytes + 64 + offset, dtype=torch.uint8, pin_memory=pinned).numpy()
    start = -raw.ctypes.data % 64 + offset
    out = raw[start:start + a.nbytes].view(np.uint8)
    out = np.ndarray(a.shape, np.float64, buffer=out.data)
    out[...] = a
    assert out.ctypes.data % 64 == offset
    return out


@pytest.mark.parametrize("prec", [gks.GKS_FP64, gks.GKS_FP32_BULK])
@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("offset", [0, 4, 8, 9])
def test_states_round_trip_from_any_address(prec, pinned, offset):
    p = wl.riemann_2d(37, 21, seed=3, mu=1e-4, Pr=0.72)
    want = [a.astype(np.float32).astype(np.float64) for a in (p.U, p.Wx, p.Wy)]
    src = [_at(a, offset, pinned) for a in want]
    s, b = gks.Solver(p, prec), gks.Batch([p, p], prec)
    gks.gks_set_state(s.h, *src, 0.5)
    gks.gks_batch_set_state(b.b, 1, *src, 0.5)
    for get in (lambda dst: gks.gks_get_state(s.h, *dst), lambda dst: gks.gks_batch_get_state(b.b, 1, *dst)[0]):
        dst = [_at(np.zeros_like(a), offset, pinned) for a in want]
        assert get(dst) == 0.5
        for x, y in zip(dst, want):
            assert np.array_equal(x, y)
    s.close()
    b.close()
