// One source's contribution to the QBX coefficients of a centre in FP64, shared
// by the all-pairs kernel (direct.cu) and the U-list kernel (fmm.cu), and the
// warp reduction of the lanes' partial coefficients.
//
// With (r, th) the polar coordinates of source - centre, W_l = H_l(k r) e^{i l th},
// q the charge, D = d k/2 and nu = e^{i phi} the unit normal,
//   alpha_l += q W_l + D (nu W_{l-1} - conj(nu) W_{l+1}).
// H_{-m} = (-1)^m H_m lets the orders +m and -m share all their products: with
// psi = th - phi, K_m = (2m/x) H_m = H_{m-1} + H_{m+1} and E_m = H_{m-1} - H_{m+1},
//   alpha_m          += A_m + i B_m,    (-1)^m alpha_{-m} += A_m - i B_m,
//   A_m = q H_m cos(m th) + D (E_m cos psi cos(m th) + K_m sin psi sin(m th)),
//   B_m = q H_m sin(m th) + D (E_m cos psi sin(m th) - K_m sin psi cos(m th)),
// whose angular factors are real. The recurrence H_{m+1} = K_m - H_{m-1} is
// linear, so it runs on q H_m and D H_m themselves and no complex product is
// left in the loop. The FP64 pipe (two lanes per clock and SM) bounds both
// kernels, so the count of FP64 instructions is what matters: 11 per order for
// a charge, 23 for a dipole, 29 for both, against 24, 32 and 40 when W_m and
// W_{-m} are formed and multiplied by q, D nu and D conj(nu) as complex numbers
// (all 16384 centres of the 8192-node starfish, p = 12, both layers, through
// the FMM: 4.04 -> 3.62 ms for the whole evaluation).
#pragma once
#include "special.cuh"

// Partial coefficients of one lane: acc[0] alpha_0, acc[2m] A_m, acc[2m + 1] B_m
// (acc[1] stays zero).
template <int PM, bool HS, bool HD>
__device__ __forceinline__ void p2qbxl_pair(cd (&acc)[2 * PM + 2], double dx, double dy, cd q,
                                            cd dk, double nx, double ny, double k, double ik,
                                            int p) {
  const double r2 = dx * dx + dy * dy;
  if (r2 == 0.0) return;  // a source on a centre has no expansion (Condition 1)
  // one reciprocal square root gives r, 1/r and 1/x (ik = 1/k): no division
  const double ir = rsqrt(r2), x = k * (r2 * ir), ix = ik * ir, ix2 = 2.0 * ix;
  const double c1 = dx * ir, s1 = dy * ir;
  cd h0, h1;
  hankel01(x, ix, h0, h1);
  cd sp, sc, dp, dc;  // q H_{m-1}, q H_m, D H_{m-1}, D H_m
  double cpsi = 0.0, spsi = 0.0;
  if (HS) {
    sp = cmul(q, h0);
    sc = cmul(q, h1);
    acc[0] = cadd(acc[0], sp);
  }
  if (HD) {
    dp = cmul(dk, h0);
    dc = cmul(dk, h1);
    cpsi = fma(c1, nx, s1 * ny);
    spsi = fma(s1, nx, -c1 * ny);
    const double t = -2.0 * cpsi;  // E_0 = -2 H_1, K_0 = 0
    acc[0].x = fma(dc.x, t, acc[0].x);
    acc[0].y = fma(dc.y, t, acc[0].y);
  }
  // (c, s) = (cos m th, sin m th); the dipole-only form turns the products
  // (ac, as) = cos psi (c, s) and (bc, bs) = sin psi (c, s) instead
  double c = c1, s = s1;
  double ac = cpsi * c1, as = cpsi * s1, bc = spsi * c1, bs = spsi * s1;
  auto turn = [&](double& u, double& v) {
    const double t = fma(u, c1, -v * s1);
    v = fma(u, s1, v * c1);
    u = t;
  };
#pragma unroll
  for (int m = 1; m <= PM; ++m) {
    if (m > p) break;
    if (m > 1) {
      if (HS) {
        turn(c, s);
        if (HD) {
          ac = cpsi * c;
          as = cpsi * s;
          bc = spsi * c;
          bs = spsi * s;
        }
      } else {
        turn(ac, as);
        turn(bc, bs);
      }
    }
    cd& A = acc[2 * m];
    cd& B = acc[2 * m + 1];
    const double cm = (double)m * ix2;
    if (HS) {
      A.x = fma(sc.x, c, A.x);
      A.y = fma(sc.y, c, A.y);
      B.x = fma(sc.x, s, B.x);
      B.y = fma(sc.y, s, B.y);
      const cd n = mk(fma(cm, sc.x, -sp.x), fma(cm, sc.y, -sp.y));
      sp = sc;
      sc = n;
    }
    if (HD) {
      const cd K = cscale(dc, cm);
      const cd n = csub(K, dp);
      const cd E = csub(dp, n);
      A.x = fma(E.x, ac, fma(K.x, bs, A.x));
      A.y = fma(E.y, ac, fma(K.y, bs, A.y));
      B.x = fma(E.x, as, fma(-K.x, bc, B.x));
      B.y = fma(E.y, as, fma(-K.y, bc, B.y));
      dp = dc;
      dc = n;
    }
  }
}

// Sums the lanes' partial coefficients over the warp by a reduce-scatter of
// shuffles (31 complex shuffles for 32 entries instead of 160 for a butterfly):
// afterwards lane L holds the sum of entry L in acc[0]. Entries 32 and 33 (order
// 16) are summed by a butterfly into x32, x33 on every lane; padding both of
// them to a second 32 would double the shuffles.
template <int NC>
__device__ __forceinline__ void warp_reduce_scatter(cd (&acc)[NC], int lane, cd& x32, cd& x33) {
  static_assert(NC <= 34, "at most order 16");
  constexpr unsigned kAll = 0xffffffffu;
  x32 = NC > 32 ? acc[NC - 2] : mk(0.0, 0.0);
  x33 = NC > 32 ? acc[NC - 1] : mk(0.0, 0.0);
  if (NC > 32) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
      x32.x += __shfl_xor_sync(kAll, x32.x, off);
      x32.y += __shfl_xor_sync(kAll, x32.y, off);
      x33.x += __shfl_xor_sync(kAll, x33.x, off);
      x33.y += __shfl_xor_sync(kAll, x33.y, off);
    }
  }
  constexpr int N = NC < 32 ? NC : 32;
#pragma unroll
  for (int h = 16; h >= 1; h >>= 1) {
    const bool upper = (lane & h) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const cd lo = i < N ? acc[i] : mk(0.0, 0.0);
      const cd hi = i + h < N ? acc[i + h] : mk(0.0, 0.0);
      const cd send = upper ? lo : hi;
      cd keep = upper ? hi : lo;
      keep.x += __shfl_xor_sync(kAll, send.x, h);
      keep.y += __shfl_xor_sync(kAll, send.y, h);
      if (i < N) acc[i] = keep;
    }
  }
}

// The coefficient(s) lane L forms from the scattered sums v (entry L), x32, x33:
// fn(l, alpha_l) for l = 0 on lane 0, l = m on lane 2m, l = -m on lane 2m + 1,
// and l = +-16 on lanes 0 and 1.
template <int PM, typename Fn>
__device__ __forceinline__ void pair_coefficients(cd v, cd x32, cd x33, int lane, int p, Fn&& fn) {
  const cd o = mk(__shfl_xor_sync(0xffffffffu, v.x, 1), __shfl_xor_sync(0xffffffffu, v.y, 1));
  const int m = lane >> 1;
  auto form = [&](cd A, cd B, int mm) {
    if ((lane & 1) == 0) return mk(A.x - B.y, A.y + B.x);      // A + i B
    const cd t = mk(A.x + B.y, A.y - B.x);                     // A - i B
    return (mm & 1) ? mk(-t.x, -t.y) : t;
  };
  if (m == 0) {
    if (lane == 0) fn(0, v);
    if (PM == 16 && p == 16) fn(lane == 0 ? 16 : -16, form(x32, x33, 16));
  } else if (m <= p) {
    fn((lane & 1) ? -m : m, (lane & 1) ? form(o, v, m) : form(v, o, m));
  }
}
