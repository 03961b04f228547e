"""Writes hankel_table_far.h: the polynomial pieces of H_0 and H_1 on
8 <= x < 32 in FP64, on intervals of width 1/2 (beyond 8 the functions oscillate
with a fixed wavelength, so equal widths need the least degree): truncated
Chebyshev series of degree 10 in t in [-1, 1] (truncation below 1e-17) written
out as monomials. Values come from mpmath at 40 digits.
Run: python gen_hankel_table_far.py > hankel_table_far.h
"""
import mpmath as mp

from gen_hankel_table import chebyshev_coefficients, to_monomial

DEGREE = 10
ROWS = 48                        # [8 + i/2, 8 + (i+1)/2)


def emit():
    fs = [lambda x: mp.besselj(0, x), lambda x: mp.bessely(0, x),
          lambda x: mp.besselj(1, x), lambda x: mp.bessely(1, x)]
    R = [[to_monomial(chebyshev_coefficients(f, 8 + mp.mpf(i) / 2, 8 + mp.mpf(i + 1) / 2, 24),
                      DEGREE) for f in fs] for i in range(ROWS)]
    lines = [
        "// Generated by gen_hankel_table_far.py (mpmath, 40 digits); do not edit.",
        "// Row i: [8 + i/2, 8 + (i+1)/2), t = 4 x - 33 - 2 i. Entry [(d * 2 + q) * kHankFarRows",
        "// + row] holds the degree-d coefficients of pair q: (J0, Y0), (J1, Y1).",
        "#pragma once",
        "constexpr int kHankFarRows = %d, kHankFarDeg = %d;" % (ROWS, DEGREE),
        "static __device__ const double2 kHankTabFar[%d] = {" % ((DEGREE + 1) * 2 * ROWS),
    ]
    for d in range(DEGREE + 1):
        for q in range(2):
            lines.append("    " + ", ".join(
                "{%s, %s}" % tuple(mp.nstr(r[2 * q + c][d], 17, min_fixed=1, max_fixed=0)
                                   for c in range(2)) for r in R) + ",")
    lines.append("};")
    return "\n".join(lines) + "\n"


if __name__ == "__main__":
    print(emit(), end="")
