"""The FP64 tables of psi, psi' and psi'' of the adjoint kernels
(csrc/lbm_psi64_table.cuh, generated by csrc/gen_psi64_table.py), parsed from
the source and evaluated as the device does (segment and midpoint from the bits
of the argument, Horner's rule), against mpmath.  No GPU needed.

Tolerance, derived: the last Horner step adds the segment's leading coefficient
and a correction of at most a twentieth of the function's scale, each rounded
once: two half-ulps, 2.2e-16, of the scale, which is psi itself (it grows by 6 %
within a segment), max(|psi'|, 1e-2 psi) and max(|psi''|, 1e-2 psi) (both fall
below FP64 resolution of psi far from a wall)."""
import os
import re

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_1603_08221_gb300", "csrc", "lbm_psi64_table.cuh")


def _table():
    src = open(SRC).read()
    body = src[src.index("kPsi64[512]"):]
    body = body[body.index("{") + 1:body.index("};")]
    return np.array([[float(v) for v in r.split(",")] for r in re.findall(r"\{([^}]*)\}", body)])


def _evaluate(T, a):
    hi = (a.view(np.uint64) >> np.uint64(32)).astype(np.int64)
    mid = ((((hi >> 15) << 15) | 0x4000).astype(np.uint64) << np.uint64(32)).view(np.float64)
    row, u = T[(hi >> 15) - ((1023 - 10) << 5)], a - mid
    out = []
    for f in range(3):
        v = row[:, 24 + f]
        for k in range(7, -1, -1):
            v = v * u + row[:, 3 * k + f]
        out.append(v)
    return out


@pytest.mark.parametrize("lo,hi", [(2.0 ** -10, 0.1), (0.1, 1.0), (1.0, 8.0), (8.0, 63.999)])
def test_tables_against_mpmath(lo, hi):
    T = _table()
    assert T.shape == (512, 28)
    edges = 2.0 ** np.arange(-10, 6) * 1.03125
    a = np.concatenate([np.geomspace(lo, hi, 400), edges[(edges >= lo) & (edges < hi)],
                        np.nextafter(edges, 0)[(edges > lo) & (edges < hi)]])
    got = _evaluate(T, a)
    with mp.workdps(40):
        for k, x in enumerate(a):
            x = mp.mpf(float(x))
            e, ex = mp.expint(1, x), mp.e ** (-x)
            psi = 1 + (x - 1) * ex - x * x * e
            for f, ref in enumerate((psi, 2 * ex - 2 * x * e, -2 * e)):
                scale = psi if f == 0 else max(abs(ref), psi / 100)
                assert abs(mp.mpf(float(got[f][k])) - ref) <= 2.3e-16 * scale, (f, float(x))
