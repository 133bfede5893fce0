"""The FP32 tables of psi and psi' that the step kernels read
(csrc/lbm_psi_table.cuh, generated by csrc/gen_psi_table.py), parsed from the
source and evaluated as the device does (segment from the bits of the
argument, cubic by fma in FP32), against scipy.  No GPU needed.

Tolerances, derived from the roundings of the evaluation: psi = min(a, 1) q
with q within a few units of 2^-24 of itself (one rounding of each of the two
leading coefficients' sum, of q0 itself and of the final product: under 3
2^-24 = 1.8e-7 relative); psi' <= 2 is not scaled: under 3 half-units of 2,
2^-23 + 2^-24 = 1.8e-7 absolute."""
import os
import re

import numpy as np
import pytest
import scipy.special

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_1603_08221_gb300", "csrc", "lbm_psi_table.cuh")
LOW = 2.0 ** -22


def _table(name):
    src = open(SRC).read()
    body = src[src.index(name + "["):]
    body = body[body.index("{") + 1:body.index("};")]
    rows = [[float(v.rstrip("f")) for v in r.split(",")] for r in re.findall(r"\{([^}]*)\}", body)]
    return np.array(rows, dtype=np.float32)


def _fma(a, b, c):
    return (a.astype(np.float64) * b + c).astype(np.float32)


def _cubic(T, a):
    am = np.minimum(a, np.float32(16))
    edge = np.maximum(am, np.float32(LOW)).view(np.uint32) & np.uint32(0xFFF80000)
    q = T[(edge >> 19).astype(int) - (105 << 4)]
    u = am - edge.view(np.float32)
    return _fma(_fma(_fma(q[:, 3], u, q[:, 2]), u, q[:, 1]), u, q[:, 0])


def _reference(a):
    """psi (from its series below 1e-3, where the closed form cancels) and psi'."""
    a = a.astype(np.float64)
    e = scipy.special.exp1(a)
    psi = 1 + (a - 1) * np.exp(-a) - a * a * e
    g = np.euler_gamma
    small = a < 1e-3
    series = (2 * a + a * a * (np.log(a) + g - 1.5) - a ** 3 / 3 + a ** 4 / 24 - a ** 5 / 180)
    return np.where(small, series, psi), 2 * np.exp(-a) - 2 * a * e


EDGES = np.concatenate([np.float32(2.0) ** np.arange(-22, 5), [1.0625, 15.999999, 16.0]])


@pytest.mark.parametrize("a", [np.geomspace(1e-12, 1e-6, 20001), np.geomspace(1e-6, 1.0, 200001),
                               np.linspace(1.0, 17.0, 200001), EDGES,
                               np.nextafter(EDGES.astype(np.float32), np.float32(0))])
def test_tables_against_scipy(a):
    a = np.asarray(a, dtype=np.float32)
    psi = _cubic(_table("kPsiTab"), a) * np.minimum(a, np.float32(1))
    dpsi = _cubic(_table("kDpsiTab"), a)
    ref, dref = _reference(a)
    assert np.abs(psi / ref - 1).max() < 3 * 2.0 ** -24
    assert np.abs(dpsi - dref).max() < 3 * 2.0 ** -24


def test_every_segment_is_there():
    for name in ("kPsiTab", "kDpsiTab"):
        assert _table(name).shape == (26 * 16 + 1, 4)
    last = [_table("kPsiTab")[-1].tolist(), _table("kDpsiTab")[-1].tolist()]
    assert last == [[1, 0, 0, 0], [0, 0, 0, 0]]
