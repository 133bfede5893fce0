"""Generates lbm_psi64_table.cuh: FP64 tables of psi (Eq. psi), psi' and psi''
for the adjoint kernels (lbm_adjoint.cu).

Segments: 32 per octave of the argument from 2^-10 to 64, picked by the
exponent and the top five mantissa bits.  In a segment with midpoint c each of
the three functions is a polynomial of degree 8 in u = a - c (exact), through
its values at the nine Chebyshev nodes in 40-digit arithmetic: the remainder is
below 1e-18 of psi.  A row holds the 27
coefficients as (psi_k, psi'_k, psi''_k), k = 0 .. 8, and one pad.

From 16 on, where the derivatives fall by e within a segment or two of an octave
(relative remainder 9e-14 on [16, 32], 4e-11 on [32, 64]), psi' and psi'' have a
table of their own with segments of a quarter, 64 and 128 in the two octaves, rows
(psi'_k, psi''_k): remainder 8e-17 of either.

    python paper_1603_08221_gb300/csrc/gen_psi64_table.py > \
        paper_1603_08221_gb300/csrc/lbm_psi64_table.cuh
"""
from __future__ import annotations

import mpmath as mp

mp.mp.dps = 40
OCTAVE0, OCTAVES, SEGS, DEG = -10, 16, 32, 8
FAR, WIDTH = 16, mp.mpf(1) / 4


def functions(a):
    e, x = mp.expint(1, a), mp.e ** (-a)
    return 1 + (a - 1) * x - a * a * e, 2 * x - 2 * a * e, -2 * e


def newton(us, fs):
    """Monomial coefficients of the polynomial through (us, fs)."""
    n = len(us)
    d = list(fs)
    for k in range(1, n):
        for i in range(n - 1, k - 1, -1):
            d[i] = (d[i] - d[i - 1]) / (us[i] - us[i - k])
    c = [mp.mpf(0)] * n
    for k in range(n - 1, -1, -1):
        c = [(-us[k] * c[i]) + (c[i - 1] if i else mp.mpf(0)) for i in range(n)]
        c[0] += d[k]
    return c


def segment(c, h):
    """Polynomials in u = a - c of psi, psi' and psi'' on [c - h / 2, c + h / 2]."""
    us = [h / 2 * mp.cos(mp.pi * (2 * k + 1) / (2 * (DEG + 1))) for k in range(DEG + 1)]
    vals = [functions(c + u) for u in us]
    return [newton(us, [v[f] for v in vals]) for f in range(3)]


def main():
    rows, far = [], []
    for o in range(OCTAVE0, OCTAVE0 + OCTAVES):
        for s in range(SEGS):
            polys = segment(mp.mpf(2) ** o * (1 + (mp.mpf(s) + mp.mpf(1) / 2) / SEGS),
                            mp.mpf(2) ** o / SEGS)
            rows.append([polys[f][k] for k in range(DEG + 1) for f in range(3)] + [mp.mpf(0)])
    for s in range(int((64 - FAR) / WIDTH)):
        polys = segment(FAR + (s + mp.mpf(1) / 2) * WIDTH, WIDTH)
        far.append([polys[f][k] for k in range(DEG + 1) for f in (1, 2)])
    print("// lbm_psi64_table.cuh - generated by gen_psi64_table.py (segments and forms there).")
    print(f"constexpr int kPsi64Octave0 = {OCTAVE0}, kPsi64Octaves = {OCTAVES}, kPsi64Row = "
          f"{3 * (DEG + 1) + 1};")
    print(f"__device__ __align__(16) const double kPsi64[{OCTAVES * SEGS}][kPsi64Row] = {{")
    for r in rows:
        print("    {" + ", ".join(mp.nstr(v, 18) for v in r) + "},")
    print("};")
    print(f"__device__ __align__(16) const double kPsi64Far[{len(far)}][{2 * (DEG + 1)}] = {{")
    for r in far:
        print("    {" + ", ".join(mp.nstr(v, 18) for v in r) + "},")
    print("};")


if __name__ == "__main__":
    main()
