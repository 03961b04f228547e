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
// whose angular factors are real. With the strengths taken into the sequences,
//   G_m = q H_m + U_{m-1} - U_{m+1},  L_m = (2m/x) V_m,  U = D cos psi H, V = D sin psi H,
//   A_m = G_m cos m th + L_m sin m th,  B_m = G_m sin m th - L_m cos m th,
// each running through the recurrence X_{m+1} = (2m/x) X_m - X_{m-1} (it is
// linear), no complex product is left in the loop. The FP64 pipe (two lanes per
// clock and SM) bounds both kernels, so the count of FP64 instructions is what
// matters: 11 per order for a charge, 21 for a dipole, 25 for both, against 24, 32
// and 40 when W_m and W_{-m} are formed and multiplied by q, D nu and D conj(nu) as
// complex numbers. (Without U and V, 11, 27 and 31: all pairs of 2048 nodes and 4096
// centres of order 12, both layers, 7.69 -> 7.01 ms; the U lists of the 8192-node
// starfish 0.39 -> 0.32 ms.)
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
  cd sp, sc, up, uc, vp, vc;  // q H, U, V at orders m - 1 and m
  if (HS) {
    sp = cmul(q, h0);
    sc = cmul(q, h1);
    acc[0] = cadd(acc[0], sp);
  }
  if (HD) {
    const cd d0 = cmul(dk, h0), d1 = cmul(dk, h1);
    const double cpsi = fma(c1, nx, s1 * ny), spsi = fma(s1, nx, -c1 * ny);
    up = cscale(d0, cpsi);
    uc = cscale(d1, cpsi);
    vp = cscale(d0, spsi);
    vc = cscale(d1, spsi);
    acc[0].x = fma(-2.0, uc.x, acc[0].x);  // U_{-1} = -U_1
    acc[0].y = fma(-2.0, uc.y, acc[0].y);
  }
  double c = c1, s = s1;  // cos m th, sin m th
#pragma unroll
  for (int m = 1; m <= PM; ++m) {
    if (m > p) break;
    if (m > 1) {
      const double t = fma(c, c1, -s * s1);
      s = fma(c, s1, s * c1);
      c = t;
    }
    cd& A = acc[2 * m];
    cd& B = acc[2 * m + 1];
    const double cm = (double)m * ix2;
    auto next = [&](cd& prev, cd& cur) {
      const cd n = mk(fma(cm, cur.x, -prev.x), fma(cm, cur.y, -prev.y));
      prev = cur;
      cur = n;
    };
    cd G;
    if (HD) {
      const cd u0 = up;
      next(up, uc);  // uc = U_{m+1}
      G = csub(u0, uc);
      if (HS) G = cadd(G, sc);
      const cd L = cscale(vc, cm);
      const cd n = csub(L, vp);
      vp = vc;
      vc = n;
      A.x = fma(G.x, c, fma(L.x, s, A.x));
      A.y = fma(G.y, c, fma(L.y, s, A.y));
      B.x = fma(G.x, s, fma(-L.x, c, B.x));
      B.y = fma(G.y, s, fma(-L.y, c, B.y));
    } else {
      G = sc;
      A.x = fma(G.x, c, A.x);
      A.y = fma(G.y, c, A.y);
      B.x = fma(G.x, s, B.x);
      B.y = fma(G.y, s, B.y);
    }
    if (HS) next(sp, sc);
  }
}

// keep += the value send of lane ^ off (complex FP64, and float-float in ff.cuh)
__device__ __forceinline__ cd lane_zero(const cd*) { return mk(0.0, 0.0); }
__device__ __forceinline__ void lane_add(cd& keep, const cd& send, int off) {
  const double x = __shfl_xor_sync(0xffffffffu, send.x, off);
  const double y = __shfl_xor_sync(0xffffffffu, send.y, off);
  keep.x += x;
  keep.y += y;
}

// Sums the partial coefficients of a group of W lanes (32, or 16: two centres per
// warp) by a reduce-scatter of shuffles (31 or 30 complex shuffles for 32 entries
// instead of 160 for a butterfly): afterwards lane g of the group holds the sums of
// entries (32 / W) g .. in acc[0..32 / W). Entries 32 and 33 (order 16) are summed by
// a butterfly into x32, x33 on every lane; padding both of them to a second 32
// would double the shuffles.
template <int W, int NC, typename V>
__device__ __forceinline__ void group_reduce_scatter(V (&acc)[NC], int lane, V& x32, V& x33) {
  static_assert(NC <= 34, "at most order 16");
  const V zero = lane_zero((const V*)nullptr);
  x32 = NC > 32 ? acc[NC - 2] : zero;
  x33 = NC > 32 ? acc[NC - 1] : zero;
  if (NC > 32) {
#pragma unroll
    for (int off = W / 2; off >= 1; off >>= 1) {
      lane_add(x32, x32, off);
      lane_add(x33, x33, off);
    }
  }
  constexpr int N = NC < 32 ? NC : 32;
#pragma unroll
  for (int h = 16; h >= 32 / W; h >>= 1) {
    const int off = h * W / 32;
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const V lo = i < N ? acc[i] : zero;
      const V hi = i + h < N ? acc[i + h] : zero;
      const V send = upper ? lo : hi;
      V keep = upper ? hi : lo;
      lane_add(keep, send, off);
      if (i < N) acc[i] = keep;
    }
  }
}

// The coefficients that lane g of the group forms from the scattered sums v0 (and
// v1 for W = 16), x32, x33: fn(l, alpha_l). W = 32: l = 0 on lane 0, l = m on lane
// 2m, l = -m on lane 2m + 1, l = +-16 on lanes 0 and 1; W = 16: l = +-g on lane g,
// l = +-16 on lane 0.
template <int W, int PM, typename Fn>
__device__ __forceinline__ void pair_coefficients(cd v0, cd v1, cd x32, cd x33, int g, int p,
                                                  Fn&& fn) {
  auto plus = [](cd A, cd B) { return mk(A.x - B.y, A.y + B.x); };  // A + i B
  auto minus = [](cd A, cd B, int m) {                              // (-1)^m (A - i B)
    const cd t = mk(A.x + B.y, A.y - B.x);
    return (m & 1) ? mk(-t.x, -t.y) : t;
  };
  if (W == 16) {
    if (g == 0) {
      fn(0, v0);
      if (PM == 16 && p == 16) {
        fn(16, plus(x32, x33));
        fn(-16, minus(x32, x33, 16));
      }
    } else if (g <= p) {
      fn(g, plus(v0, v1));
      fn(-g, minus(v0, v1, g));
    }
    return;
  }
  const cd o = mk(__shfl_xor_sync(0xffffffffu, v0.x, 1), __shfl_xor_sync(0xffffffffu, v0.y, 1));
  const int m = g >> 1;
  if (m == 0) {
    if (g == 0) fn(0, v0);
    if (PM == 16 && p == 16) fn(g == 0 ? 16 : -16, g == 0 ? plus(x32, x33) : minus(x32, x33, 16));
  } else if (m <= p) {
    fn((g & 1) ? -m : m, (g & 1) ? minus(o, v0, m) : plus(v0, o));
  }
}
