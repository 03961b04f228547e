"""Writes hankel_table_ff.h: the polynomial pieces of H_0 = J_0 + i Y_0 and
H_1 = J_1 + i Y_1 that the float-float (pair of FP32) kernels of the mixed path
evaluate on 2^-16 <= x < 32.

* 2^-16 <= x < 8: eight intervals per octave as in gen_hankel_table.py (the
  interval index is a bit field of x; the singularity at 0 lies 17 half-widths
  from every centre).
* 8 <= x < 32: intervals of width 1/2 (beyond 8 the functions oscillate with a
  fixed wavelength and a geometric partition would need a higher degree).

On each interval the four functions are truncated Chebyshev series of degree 9
in t in [-1, 1] (truncation below 2e-15 of |H_0|, |H_1|) written out as
monomials. The coefficients of degree j shrink like 17^-j, so FP32 coefficients
serve the upper degrees; the lowest kHankLoFf carry a second FP32 part (value
minus its FP32 rounding). Values come from mpmath at 40 digits.
Run: python gen_hankel_table_ff.py > hankel_table_ff.h
"""
import mpmath as mp
import numpy as np

from gen_hankel_table import chebyshev_coefficients, to_monomial

DEGREE, LO = 9, 6
OCTAVES = tuple(range(-16, 3))
UNIFORM = tuple(range(48))       # [8 + i/2, 8 + (i+1)/2)


def intervals():
    for E in OCTAVES:
        for j in range(8):
            a = mp.mpf(2) ** E * (1 + mp.mpf(j) / 8)
            yield a, a + mp.mpf(2) ** E / 8
    for i in UNIFORM:
        yield 8 + mp.mpf(i) / 2, 8 + mp.mpf(i + 1) / 2


def split(v):
    """v as an FP32 value and the FP32 rounding of what it leaves."""
    hi = np.float32(float(v))
    lo = np.float32(float(v - mp.mpf(float(hi))))
    return "%.9gf" % hi if "." in "%.9g" % hi or "e" in "%.9g" % hi else "%.9g.f" % hi, \
        "%.9gf" % lo if "." in "%.9g" % lo or "e" in "%.9g" % lo else "%.9g.f" % lo


def emit():
    fs = [lambda x: mp.besselj(0, x), lambda x: mp.bessely(0, x),
          lambda x: mp.besselj(1, x), lambda x: mp.bessely(1, x)]
    R = [[to_monomial(chebyshev_coefficients(f, a, b, 20), DEGREE) for f in fs]
         for a, b in intervals()]
    n = len(R)
    lines = [
        "// Generated by gen_hankel_table_ff.py (mpmath, 40 digits); do not edit.",
        "// Rows 0..%d: [2^E (1 + j/8), 2^E (1 + (j+1)/8)), E = %d..%d, t = 16 x / 2^E - 17 - 2 j;"
        % (8 * len(OCTAVES) - 1, OCTAVES[0], OCTAVES[-1]),
        "// rows %d..%d: [8 + i/2, 8 + (i+1)/2), t = 4 x - 33 - 2 i. Entry [(d * 2 + q) *"
        % (8 * len(OCTAVES), n - 1),
        "// kHankRowsFf + row] holds the degree-d coefficients of pair q: (J0, Y0), (J1, Y1);",
        "// kHankLoFf: the same entries' second parts, d < kHankLoFf.",
        "#pragma once",
        "constexpr int kHankRowsFf = %d, kHankMinExpFf = %d, kHankUniformFf = %d;" % (
            n, OCTAVES[0], 8 * len(OCTAVES)),
        "constexpr int kHankDegFf = %d, kHankLoFf = %d;" % (DEGREE, LO),
    ]
    for part, name, deg in ((0, "kHankTabFf", DEGREE + 1), (1, "kHankTabFfLo", LO)):
        lines.append("static __device__ const float2 %s[%d] = {" % (name, deg * 2 * n))
        for d in range(deg):
            for q in range(2):
                lines.append("    " + ", ".join(
                    "{%s, %s}" % (split(r[2 * q][d])[part], split(r[2 * q + 1][d])[part])
                    for r in R) + ",")
        lines.append("};")
    return "\n".join(lines) + "\n"


if __name__ == "__main__":
    print(emit(), end="")
