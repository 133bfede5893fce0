"""Generates lbm_psi_table.cuh: the FP32 tables of psi (Eq. psi) and psi' that
the step kernels read.

Segments: 16 per octave of the argument from 2^-22 to 16, so that a segment
is picked by the exponent and the top four mantissa bits.  In a segment with
left edge c, with u = a - c (exact in FP32),

  psi(a) = min(a, 1) (q0 + q1 u + q2 u^2 + q3 u^3),
  psi'(a) =           q0 + q1 u + q2 u^2 + q3 u^3,

the cubic interpolating at the four Chebyshev nodes of the segment in
40-digit arithmetic.  psi / min(a, 1) is of order one everywhere (2 at
a = 0), so the relative error is that of FP32 however small the argument.
The first segment reaches down to a = 0, the last entry holds the values from
a = 16 on (1 and 0: 1 - psi(16) < 2^-25).

    python paper_1603_08221_gb300/csrc/gen_psi_table.py > \
        paper_1603_08221_gb300/csrc/lbm_psi_table.cuh
"""
from __future__ import annotations

import mpmath as mp

mp.mp.dps = 40
OCTAVE0, OCTAVES, SEGS = -22, 26, 16


def E1(a):
    return mp.expint(1, a)


def psi(a):
    return 1 + (a - 1) * mp.e ** (-a) - a * a * E1(a)


def scaled(a):
    return psi(a) / min(a, mp.mpf(1))


def dpsi(a):
    return 2 * mp.e ** (-a) - 2 * a * E1(a)


def cubic(f, c, lo, hi):
    """Coefficients in u = a - c of the cubic through f at the Chebyshev
    nodes of [lo, hi]."""
    nodes = [(lo + hi) / 2 + (hi - lo) / 2 * mp.cos(mp.pi * (2 * k + 1) / 8) for k in range(4)]
    A = mp.matrix(4, 4)
    b = mp.matrix(4, 1)
    for r, a in enumerate(nodes):
        for k in range(4):
            A[r, k] = (a - c) ** k
        b[r] = f(a)
    return list(mp.lu_solve(A, b))


def table(f, last):
    rows = []
    for o in range(OCTAVE0, OCTAVE0 + OCTAVES):
        for s in range(SEGS):
            c = mp.mpf(2) ** o * (1 + mp.mpf(s) / SEGS)
            h = mp.mpf(2) ** o / SEGS
            rows.append(cubic(f, c, mp.mpf(0) if not rows else c, c + h))
    rows.append([mp.mpf(last), mp.mpf(0), mp.mpf(0), mp.mpf(0)])
    return rows


def emit(name, rows):
    print(f"__device__ const float4 {name}[PSI_SEGMENTS] = {{")
    for r in rows:
        print("    {" + ", ".join(f"{float(v):.9e}f" for v in r) + "},")
    print("};")


def main():
    print("// lbm_psi_table.cuh - generated by gen_psi_table.py (segments and forms there).")
    print(f"constexpr int PSI_SEGMENTS = {OCTAVES * SEGS + 1};")
    emit("kPsiTab", table(scaled, 1))
    emit("kDpsiTab", table(dpsi, 0))


if __name__ == "__main__":
    main()
