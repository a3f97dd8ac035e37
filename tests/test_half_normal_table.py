"""The nodes and polynomials of the FP64 erfc / exp table (csrc/gks_half_normal.cuh), on the CPU, against the C
library's functions: every node, and a dense sweep of the evaluation as the device does it, in relative terms."""
import math
import os
import re
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _nodes():
    src = open(os.path.join(ROOT, "paper_1412_4489_gb300", "csrc", "gks_half_normal.cuh")).read()
    body = src[src.index("kHalfNode[kHalfNodes] = {"):src.index("struct alignas(16) HalfTable")]
    pairs = re.findall(r"\{([0-9.e+-]+), ([0-9.e+-]+)\}", body)
    assert len(pairs) == 193 and "kHalfNodes = 193, kHalfDegree = 10" in src
    return [(float(a), float(b)) for a, b in pairs]


def test_every_node():
    """The C library's erfc and exp round to about one unit each, the nodes to half a unit."""
    for k, (h, g) in enumerate(_nodes()):
        z = k / 32.0
        assert abs(h - 0.5 * math.erfc(z)) <= 4 * 2.0 ** -53 * h, k
        assert abs(g - math.exp(-z * z)) <= 4 * 2.0 ** -53 * g, k  # z * z is exact


def _rows():
    """Taylor coefficients of erfc(z) / 2 about the nodes, as half_table() forms them."""
    out = []
    for k, (h, g) in enumerate(_nodes()):
        z, e = k / 32.0, -0.56418958354775628 * g
        h0, h1, f, row = 1.0, 2.0 * z, 1.0, [h]
        for n in range(10):
            f /= n + 1
            row.append((-h0 if n & 1 else h0) * f * e)
            h0, h1 = h1, 2.0 * z * h1 - 2.0 * (n + 1) * h0
        out.append(row)
    return np.array(out)


def _evaluate(rows, z):
    big = 211106232532992.0
    m = z + big
    d = z - (m - big)
    k = ((m - big) * 32.0).astype(int)
    c = rows[k]
    p, q = c[:, 10].copy(), c[:, 10].copy()
    p = p * d + c[:, 9]
    for n in range(8, -1, -1):
        q = q * d + p
        p = p * d + c[:, n]
    return p, -1.7724538509055160 * q


@pytest.mark.parametrize("lo,hi", [(0.0, 1.0), (1.0, 3.0), (3.0, 5.0), (5.0, 6.0)])
def test_dense_sweep(lo, hi):
    """Relative error: the truncation after degree 10 (9 for exp), (2 z / 64)^n / n! of the value at its worst, where the
    values fall as exp(-z^2), and some roundings (the Horner sums, and the coefficients' own of up to n steps)."""
    z = np.linspace(lo, hi, 20001)[:-1]
    z = np.concatenate([z, np.arange(lo, hi, 1 / 64), np.nextafter(np.arange(lo, hi, 1 / 64), 9.0)])
    t, e = _evaluate(_rows(), z)
    x = 2.0 * (hi + 1 / 64) / 64
    trunc = lambda n: 1.5 * x ** n / math.factorial(n)  # noqa: E731
    rounding = 32 * 2.0 ** -53
    for v, w in zip((t, e), (np.array([0.5 * math.erfc(a) for a in z]), np.array([math.exp(-float(Fraction(a) ** 2)) for a in z]))):
        tol = rounding + trunc(11 if v is t else 10)
        # exp's own argument is rounded: z^2 2^-53
        assert np.max(np.abs(v / w - 1.0)) <= tol + hi * hi * 2.0 ** -53
    assert np.max(np.abs(t - [0.5 * math.erfc(a) for a in z])) < 1e-15
