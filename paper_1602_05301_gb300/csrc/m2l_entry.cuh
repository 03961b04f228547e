// Entries of the sigma-normalised M2L operator of one (level, offset class),
//     T[n][lo] = sig_lo sig_n (-1)^lo W_{n+lo}(D) s^-|n+lo| (scale factors of
//     the level's power-scaled Hankel table What_m = s^|m| W_m(D)),
// computed in FP64 through the logarithms of the scale factors (the table entries
// reach 1e155, the sigma products are tiny): of order one or smaller for every n, lo. Used by
// the FP32 M2L of the mixed path and by the tensor-core M2L of the FP64 path.
#pragma once
#include "qbx_internal.h"

struct M2lNorm {
  const cd* w;       // What_m at w[m], |m| <= 2 pbmax
  const double* sg;  // log sig_j of the level
  double ls;         // log s of the level
  bool used;         // the class is a V-list offset (max(|dx|, |dy|) >= 2)
  __device__ M2lNorm(const cd* t_m2l, const double* scale, const double* lsig, int l, int cls,
                     int pbmax)
      : w(t_m2l + ((size_t)l * 49 + cls) * (4 * pbmax + 1) + 2 * pbmax),
        sg(lsig + (size_t)l * (pbmax + 1)),
        ls(log(scale[l])) {
    const int dx = cls / 7 - 3, dy = cls % 7 - 3;
    used = max(abs(dx), abs(dy)) >= 2;
  }
  // the factor is at most 1 / |What|, so it may underflow where the product does
  // not: its square root is applied twice. Orders |n + lo| > 170 of boxes below a
  // wavelength leave FP64's range in What; such an entry multiplies and makes
  // coefficients below 0.71^|n| and 0.71^|lo| (a box's own points are that near), less
  // than 1e-25 of a potential: zero
  __device__ cd entry(int n, int lo) const {
    if (!used) return mk(0.0, 0.0);
    const cd v = w[n + lo];
    if (!isfinite(v.x) || !isfinite(v.y)) return mk(0.0, 0.0);
    const double lf = sg[abs(lo)] + sg[abs(n)] - abs(n + lo) * ls;
    double f = lf < -1400.0 ? 0.0 : exp(0.5 * lf);
    const double g = (lo & 1) ? -f : f;
    return mk(v.x * f * g, v.y * f * g);
  }
};
