// Float-float arithmetic: a value as the unevaluated sum h + l of two FP32
// numbers, about 47 significant bits. GB300 runs 64 FP32 FMAs in the time of
// one FP64 FMA, and a float-float multiply-add takes about a dozen FP32
// instructions, so the mixed path's recurrences (whose results are rounded to
// FP32 and whose FP64 form was bound by the FP64 pipe) run several times
// faster in this form. Error-free transformations after Dekker (Numer. Math.
// 18, 1971) and Knuth; the compiler contracts nothing here because every
// rounding is spelled out with the _rn intrinsics.
//
// Also H_0, H_1 from the tables of hankel_table_ff.h in float-float.
#pragma once
#include <cmath>

#include "special.cuh"
#include "hankel_table_ff.h"

struct ff {
  float h, l;
};

__device__ __forceinline__ ff mkff(float h, float l) { ff r; r.h = h; r.l = l; return r; }
// s + e = a + b exactly
__device__ __forceinline__ ff two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float t = __fsub_rn(s, a);
  return mkff(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t)));
}
// the same for |a| >= |b| or a == 0
__device__ __forceinline__ ff fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return mkff(s, __fsub_rn(b, __fsub_rn(s, a)));
}
// a b with the low part not yet added in: h = fl(a.h b.h), l = the rest
__device__ __forceinline__ ff ff_mul_raw(ff a, ff b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  return mkff(p, __fmaf_rn(a.l, b.h, e));
}
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const ff p = ff_mul_raw(a, b);
  return fast_two_sum(p.h, p.l);
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  const ff s = two_sum(a.h, b.h);
  return fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
// a - b without the final renormalisation: |l| stays within a few ulp of the
// larger operand, which the products above carry along
__device__ __forceinline__ ff ff_sub_raw(ff a, ff b) {
  const ff s = two_sum(a.h, -b.h);
  return mkff(s.h, __fadd_rn(s.l, __fsub_rn(a.l, b.l)));
}
__device__ __forceinline__ float ff_f32(ff a) { return __fadd_rn(a.h, a.l); }
__device__ __forceinline__ double ff_f64(ff a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ ff ff_scale(ff a, float s) {  // s a power of two
  return mkff(__fmul_rn(a.h, s), __fmul_rn(a.l, s));
}

// v 2^sh as float-float with integer instructions only (a conversion would
// occupy the FP64 pipe): h is the leading 24 bits of v truncated, l the next
// 23. off = 896 - sh. Magnitudes outside FP32's normal range become zero (below)
// or infinity (above); l is zero where it would be subnormal.
__device__ __forceinline__ ff ff_from_f64(double v, int off) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned sgn = hi & 0x80000000u;
  // exponent field e64 - 896 + sh over the top 23 mantissa bits
  const unsigned b = __funnelshift_l(lo, hi, 3) - ((unsigned)off << 23);
  const int e = (int)((hi >> 20) & 0x7FFu) - off;
  const unsigned eb = (b & 0x7F800000u) - (23u << 23);
  const float one = __uint_as_float(eb | sgn);
  const float rest = __uint_as_float(eb | sgn | ((lo & 0x1FFFFFFFu) >> 6));
  ff r;
  r.h = __uint_as_float(sgn | (e <= 0 ? 0u : e >= 255 ? 0x7F800000u : b));
  r.l = (e <= 24 || e >= 255) ? 0.f : __fsub_rn(rest, one);
  return r;
}
// ff_from_f64 that keeps a NaN (which it makes infinite): coefficients, once each
__device__ __forceinline__ ff ff_from_f64_nan(double v, int off) {
  return ((unsigned)__double2hiint(v) & 0x7FF00000u) != 0x7FF00000u ? ff_from_f64(v, off)
                                                                    : mkff(f32_from_f64(v), 0.f);
}
// FP64 constant (any magnitude FP32 holds) as float-float, for kernel arguments
// and per-thread set-up
__device__ __forceinline__ ff ff_round(double v) {
  const float h = (float)v;
  return mkff(h, (float)(v - (double)h));
}

// 1 / sqrt(a): one Newton step from the hardware estimate, the residual formed
// exactly; relative error below 2^-44
__device__ __forceinline__ ff ff_rsqrt(ff a) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a.h));
  const float q = __fmul_rn(y, y), qe = __fmaf_rn(y, y, -q);
  float s = __fmaf_rn(-a.h, q, 1.0f);
  s = __fmaf_rn(-a.h, qe, s);
  s = __fmaf_rn(-a.l, q, s);
  // y (1 + s/2 + 3 s^2 / 8)
  return mkff(y, __fmul_rn(y, __fmul_rn(s, __fmaf_rn(0.375f, s, 0.5f))));
}

// One Horner step c + t p in float-float, c = (ch, cl).
__device__ __forceinline__ ff ff_horner(ff p, ff t, float ch, float cl) {
  const ff m = ff_mul_raw(p, t);
  const ff s = two_sum(ch, m.h);
  return mkff(s.h, __fadd_rn(s.l, __fadd_rn(m.l, cl)));
}

struct ffh {  // a complex float-float value
  ff x, y;
};
// keep += the value send of lane ^ off, not renormalised (group_reduce_scatter)
__device__ __forceinline__ ffh lane_zero(const ffh*) {
  ffh z;
  z.x = z.y = mkff(0.f, 0.f);
  return z;
}
__device__ __forceinline__ void lane_add(ff& keep, ff send, int off) {
  const float h = __shfl_xor_sync(0xffffffffu, send.h, off);
  const float l = __shfl_xor_sync(0xffffffffu, send.l, off);
  const ff s = two_sum(keep.h, h);
  keep = mkff(s.h, __fadd_rn(s.l, __fadd_rn(keep.l, l)));
}
__device__ __forceinline__ void lane_add(ffh& keep, const ffh& send, int off) {
  lane_add(keep.x, send.x, off);
  lane_add(keep.y, send.y, off);
}

// H_0, H_1 at 2^-16 <= x < 32 (x normalised) from the tables: the degrees
// kHankDegFf .. ND in FP32, the lowest ND in float-float. The coefficients
// shrink like 17^-j (0.25^j / j! where H oscillates, beyond x = 1), which bounds
// the FP32 part. Measured against mpmath at 4500 points, largest error of |H_0| and
// |H_1|: 1.5e-11 (1.9e-10 beyond x = 1) at ND = 3, 6e-15 (2.7e-14) at ND = 6.
// Results are not renormalised (ff_sub_raw).
template <int ND, bool NEED0, bool NEED1>
__device__ __forceinline__ void hankel01_ff(ff x, ffh& h0, ffh& h1) {
  static_assert(ND <= kHankLoFf, "second parts are stored for the lowest degrees");
  const unsigned bits = __float_as_uint(x.h);
  const bool low = x.h < 8.0f;
  const int ej = (int)(bits >> 20) - ((127 + kHankMinExpFf) << 3);  // 8 (E + 16) + j
  const int iu = __float2int_rd(__fmaf_rn(2.0f, x.h, -16.0f));
  int row = low ? ej : kHankUniformFf + iu;
  row = min(max(row, 0), kHankRowsFf - 1);
  // t = 16 x / 2^E - 17 - 2 j, or 4 x - 33 - 2 i: the FMA is exact in h. The second
  // part reaches 2^-18: the FP32 degrees take the sum, and where products of second
  // parts matter (2^-42 at each float-float degree) t is renormalised
  const float a = low ? __uint_as_float((258u << 23) - (bits & 0x7F800000u)) : 4.0f;
  const float b = (float)(low ? -17 - 2 * (ej & 7) : -33 - 2 * iu);
  ff t = mkff(__fmaf_rn(x.h, a, b), __fmul_rn(x.l, a));
  if (ND > 3) t = two_sum(t.h, t.l);
  const float tf = ND > 3 ? t.h : __fadd_rn(t.h, t.l);
  const float2* tb = kHankTabFf + row;
  const float2* tl = kHankTabFfLo + row;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    if (q == 0 ? !NEED0 : !NEED1) continue;
    float2 c = tb[(2 * kHankDegFf + q) * kHankRowsFf];
#pragma unroll
    for (int d = kHankDegFf - 1; d >= ND; --d) {
      const float2 k = tb[(2 * d + q) * kHankRowsFf];
      c = make_float2(__fmaf_rn(c.x, tf, k.x), __fmaf_rn(c.y, tf, k.y));
    }
    ff re = mkff(c.x, 0.f), im = mkff(c.y, 0.f);
#pragma unroll
    for (int d = ND - 1; d >= 0; --d) {
      const float2 k = tb[(2 * d + q) * kHankRowsFf], kl = tl[(2 * d + q) * kHankRowsFf];
      re = ff_horner(re, t, k.x, kl.x);
      im = ff_horner(im, t, k.y, kl.y);
    }
    if (q == 0) { h0.x = re; h0.y = im; } else { h1.x = re; h1.y = im; }
  }
}

// Arguments outside the float-float tables: FP64, out of line (rare).
static __device__ __noinline__ void hankel01_outside(double x, double* h) {
  cd h0, h1;
  hankel01_wide(x, 1.0 / x, h0, h1);
  h[0] = h0.x;
  h[1] = h0.y;
  h[2] = h1.x;
  h[3] = h1.y;
}
template <int ND, bool NEED0 = true, bool NEED1 = true>
__device__ __forceinline__ void hankel01_ff_any(ff x, ffh& h0, ffh& h1) {
  if (x.h >= 0x1p-16f && x.h < 31.99f) {
    hankel01_ff<ND, NEED0, NEED1>(x, h0, h1);
    return;
  }
  double h[4];
  hankel01_outside(ff_f64(x), h);
  if (NEED0) { h0.x = ff_round(h[0]); h0.y = ff_round(h[1]); }
  if (NEED1) { h1.x = ff_round(h[2]); h1.y = ff_round(h[3]); }
}

// Lengths in the float-float kernels are in units of 2^-sh (sh = floor(log2 k)), so
// that the wavenumber is kk in [1, 2) and every quantity of order x = k r: off =
// 896 - sh is ff_from_f64's offset. Made on the host and passed to the kernels (a
// thread forming it spends two dozen FP64 instructions).
struct FfUnits {
  int off;
  ff kk, ik2;  // kk and 2 / kk
};
inline FfUnits make_ff_units(double k) {
  auto round2 = [](double v) {
    ff r;
    r.h = (float)v;
    r.l = (float)(v - (double)r.h);
    return r;
  };
  FfUnits U;
  const int sh = std::ilogb(k);
  const double q = std::ldexp(k, -sh);
  U.off = 896 - sh;
  U.kk = round2(q);
  U.ik2 = round2(2.0 / q);
  return U;
}

// (x, y) = a displacement in those units; z = k r, ir = 1 / r and the direction
// e^{i th} in FP32. False at r = 0 (both components below FP32's normal range).
// Where r^2 or its second part would leave that range, r is formed at 2^64 times
// the size (rsqrt.approx.ftz is infinite at a subnormal square). Components below
// 2^-102 have no second part.
struct FfPolar {
  ff x, y, ir, z;  // z = k r
  float c, s;
  __device__ __forceinline__ bool set(double dx, double dy, const FfUnits& U) {
    x = ff_from_f64(dx, U.off);
    y = ff_from_f64(dy, U.off);
    ff d2 = ff_add(ff_mul_raw(x, x), ff_mul_raw(y, y));
    if (d2.h < 0x1p-76f) {
      if (x.h == 0.f && y.h == 0.f) return false;
      const ff xs = ff_scale(x, 0x1p64f), ys = ff_scale(y, 0x1p64f);
      d2 = ff_add(ff_mul_raw(xs, xs), ff_mul_raw(ys, ys));
      ir = ff_rsqrt(d2);
      z = ff_scale(ff_mul(ff_mul_raw(d2, ir), U.kk), 0x1p-64f);
      ir = ff_scale(ir, 0x1p64f);
    } else {
      ir = ff_rsqrt(d2);
      z = ff_mul(ff_mul_raw(d2, ir), U.kk);
    }
    const float irf = ff_f32(ir);
    c = ff_f32(x) * irf;
    s = ff_f32(y) * irf;
    return true;
  }
};

// a = ah + al with ah on 17 bits, so that m ah is exact for 0 <= m < 128
__device__ __forceinline__ ff split17(ff a) {
  const ff n = fast_two_sum(a.h, a.l);
  const float h = __uint_as_float(__float_as_uint(n.h) & 0xFFFFFF80u);
  return mkff(h, __fadd_rn(__fsub_rn(n.h, h), n.l));
}

// (a + i b) *= c + i d
__device__ __forceinline__ void ff_turn(ff& a, ff& b, ff c, ff d) {
  const ff t = ff_sub_raw(ff_mul_raw(a, c), ff_mul_raw(b, d));
  const ff u = ff_add(ff_mul_raw(a, d), ff_mul_raw(b, c));
  a = fast_two_sum(t.h, t.l);
  b = u;
}

// Miller's backward recurrence on f_j ~ 2^{-s j} J_j(k r), j = 0..M, kept in row
// (h, l); returns 1 / norm:
//   f_{n-1} = (2 n 2^s / x) f_n - 4^s f_{n+1},  norm = f_0 + 2 4^s (f_2 + 4^s (f_4 + ...)).
// Where f outgrows its range it is scaled by kMillerDown, and the order at which that
// happened is marked in the row (the lowest bit of l): ff_miller_value, called for j =
// 0, 1, ... M in this order, gives 2^{-s j} J_j / inv. (Scaling the stored orders at
// once, a loop over them, was over half of the fill's instructions: the lanes of a
// warp outgrow the range at different orders.)
constexpr float kMillerDown = 0x1p-60f;
__device__ __forceinline__ ff ff_miller_value(float2 v, float& scale) {
  if (__float_as_uint(v.y) & 1u) scale *= kMillerDown;
  return mkff(v.x * scale, v.y * scale);
}
__device__ __forceinline__ ff ff_miller_row(float2* row, int M, int s, const FfPolar& D,
                                            const FfUnits& U) {
  const float sg2 = pow2f(2 * s);
  ff c2 = ff_mul_raw(ff_scale(U.ik2, pow2f(s)), D.ir);  // 2 2^s / x
  c2 = fast_two_sum(c2.h, c2.l);
  const int N = miller_start_f32(M, D.z.h);  // N > M + 1
  ff f1 = mkff(0.f, 0.f), f0 = mkff(0x1p-40f, 0.f), sum = f1;
  float fn = (float)N;
  for (int nn = N; nn >= 1; --nn) {
    if ((nn & 1) == 0) sum = ff_add(f0, ff_scale(sum, sg2));
    const float ch = __fmul_rn(fn, c2.h);
    const ff cn = mkff(ch, __fmaf_rn(fn, c2.l, __fmaf_rn(fn, c2.h, -ch)));
    const ff f = ff_sub_raw(ff_mul_raw(cn, f0), ff_scale(f1, sg2));
    f1 = f0;
    f0 = fast_two_sum(f.h, f.l);
    fn -= 1.f;
    const bool over = fabsf(f0.h) >= 0x1p20f;
    if (nn - 1 <= M)
      row[nn - 1] = make_float2(
          f0.h, __uint_as_float((__float_as_uint(f0.l) & ~1u) | (over ? 1u : 0u)));
    if (over) {
      f0 = ff_scale(f0, kMillerDown);
      f1 = ff_scale(f1, kMillerDown);
      sum = ff_scale(sum, kMillerDown);
    }
  }
  const ff norm = ff_add(f0, ff_scale(sum, 2.f * sg2));
  const float r = 1.0f / norm.h;  // 1 / norm by one Newton step
  return mkff(r, __fmul_rn(r, __fmaf_rn(-norm.l, r, __fmaf_rn(-norm.h, r, 1.0f))));
}
