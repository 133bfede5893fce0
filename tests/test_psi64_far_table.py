"""The FP64 table of psi' and psi'' for arguments from 16 on (csrc/
lbm_psi64_table.cuh), parsed from the source and evaluated as the device does,
against mpmath, relative to the derivatives themselves.  No GPU needed.

Tolerance, derived: the remainder of the polynomial is (1/8)^9 / (9! 2^8) =
8e-17 of the function, which falls by a factor e per unit; its leading
coefficient is rounded once (1.1e-16), the last sum once (1.2e-16, the segment's
end lies an eighth off its middle), the correction, an eighth of it, by 2.2e-16 of
itself: 3.4e-16."""
import os
import re

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_1603_08221_gb300", "csrc", "lbm_psi64_table.cuh")


def _table():
    src = open(SRC).read()
    body = src[src.index("kPsi64Far["):]
    body = body[body.index("{") + 1:body.index("};")]
    return np.array([[float(v) for v in r.split(",")] for r in re.findall(r"\{([^}]*)\}", body)])


def _evaluate(T, a):
    hi = (a.view(np.uint64) >> np.uint64(32)).astype(np.int64)
    above = (hi >= 0x40400000).astype(np.int64)
    shift = 14 - above
    mid = ((hi >> shift) << shift) | (1 << (shift - 1))
    row = T[((hi & 0xFFFFF) >> shift) + 64 * above]
    u = a - (mid.astype(np.uint64) << np.uint64(32)).view(np.float64)
    assert np.abs(u).max() <= 0.125
    out = []
    for f in range(2):
        v = row[:, 16 + f]
        for k in range(7, -1, -1):
            v = v * u + row[:, 2 * k + f]
        out.append(v)
    return out


def test_derivatives_relative_to_themselves():
    T = _table()
    assert T.shape == (192, 18)
    edges = np.arange(16.0, 64.0, 0.25)
    a = np.concatenate([np.linspace(16, 63.999, 700), edges, np.nextafter(edges[1:], 0), [31.999999]])
    got = _evaluate(T, a)
    with mp.workdps(40):
        for k, x in enumerate(a):
            x = mp.mpf(float(x))
            e, ex = mp.expint(1, x), mp.e ** (-x)
            for f, ref in enumerate((2 * ex - 2 * x * e, -2 * e)):
                assert abs(mp.mpf(float(got[f][k])) / ref - 1) <= 3.4e-16, (f, float(x))
