// FMM-accelerated Global QBX (Sec. 7.2, Stages 2-8), FP64.
//
// Expansions about box centres, with per-level scale s = min(1, k * side):
//   multipole  phi(x) = sum_n  mh_n s^|n| W_n(x - m)            (H-expansion)
//   local      psi(x) = sum_n  lh_n s^-|n| conj(V_n(x - m))      (J-expansion)
// where W_n(z) = H_n(k|z|) e^{i n arg z} and V_n(z) = J_n(k|z|) e^{i n arg z}.
// Storing mh = a / s^|n| and lh = gamma s^|n| keeps the stored numbers of
// order one although H_n grows and J_n decays factorially with n for small
// k*side. The operators come from Graf's addition theorem (DLMF 10.23.7):
//   W_n(A - B) = sum_l W_{n+l}(A) conj(V_l(B))   (|B| < |A|),
//   V_n(A - B) = sum_l V_{n+l}(A) conj(V_l(B))   (all A, B),
// giving, in unscaled form (d the translation vector),
//   P2M   a_n     = sum_j q_j conj(V_n(y_j - m))                   (Stage 2)
//   M2M   a_s     = sum_n a'_n conj(V_{s-n}(m' - m))               (Stage 2)
//   M2L   gamma_l = (-1)^l sum_n a_n W_{n+l}(m_b - m_c)            (Stage 4)
//   P2L   gamma_l = sum_j q_j W_l(y_j - m)                         (Stage 6)
//   L2L   gamma'_s = sum_n gamma_n (-1)^{s-n} V_{s-n}(m' - m)      (Stage 7)
// and the QBX steps marked "New" in the paper: P2QBXL (Stage 3), M2QBXL
// (Stage 5) and L2QBXL (Stage 8) are P2L, M2L and L2L with a QBX centre as the
// target and order p. A double-layer source contributes
// (k/2)(nu Z_{n-1} - conj(nu) Z_{n+1}) for Z = W, and the conjugate form for
// conj(V), with nu = n_x + i n_y its normal (normal derivative of the Graf
// kernel in the source).
#include <algorithm>
#include <cstdio>
#include <mutex>
#include <set>
#include <type_traits>
#include <vector>

#include "f32x2.cuh"
#include "ff.cuh"
#include "p2qbxl_pair.cuh"
#include "tree.cuh"

namespace {

constexpr int kThreads = 128;
// Sources per shared-memory chunk in P2M / P2L. Their rows (one FP64 recurrence
// per source) are built by threads 0..kChunk-1, a full warp: the SM's FP64
// rate is shared by its warps and a warp instruction costs the same with few
// lanes active, so partly filled warps waste it (measured).
constexpr int kChunk = 32;
// Leaves holding a centre are at least this many expansion radii wide.
constexpr double kLeafOverRadius = 4.0;
// A W-list box c is translated to a centre z (M2QBXL) only if
// (R_c + r_z) <= kW * |z - m_c| (R_c: half-diagonal of c, r_z: disk radius);
// otherwise its sources are summed directly into the coefficients.
constexpr double kW = 0.6;

inline unsigned nblk(int64_t n, int b) { return (unsigned)std::max<int64_t>(1, (n + b - 1) / b); }
// opt-in shared memory per block of the current device (set by configure_kernels)
int g_smem_optin = 48 * 1024;
#define TRY_MIXED(x)                    \
  do {                                  \
    qbx_status s_ = (x);                \
    if (s_ != QBX_OK) return s_;        \
  } while (0)

struct Fmm {
  // boxes
  const int* level;
  const int* child;
  const double2* centre;
  const int2* rsrc;
  const int2* rctr;
  const int2* rtgt;
  // lists
  const int *uoff, *uidx, *voff, *vidx, *vcls, *woff, *widx, *xoff, *xidx;
  // sorted particles
  const double2* sxy;
  const double2* snrm;
  const cd* qs;
  const cd* ds;
  const float2* q32;     // FP32 charges (mixed path)
  const float4* ab32;    // FP32 dipole factors (A, B) (mixed path)
  const float4* dn32;    // FP32 (d k/2, nu) (mixed path)
  const float4 *qf, *df, *nf;  // float-float charges, d k and normals (mixed P2P)
  const int* sexp;       // e: the strengths carry 2^-e (mixed path)
  const double2* cxy;
  const double* crad;    // sorted centre radii
  const int* cid;
  const double2* txy;
  const int* tid;
  const int* tassoc;
  // orders and tables (box order pb_l per level; Q_l = 2 pb_l + 1 coefficients)
  const int* lpb;        // [n_levels]
  const long long* eoff; // [n_boxes] first coefficient of each box in mpole / local
  const double* scale;   // [n_levels]
  const double* pw;      // [n_levels][2 pbmax + 3] s^j
  const double* ipw;     // [n_levels][pbmax + 2]  s^-j
  const cd* t_m2l;       // [n_levels][49][4 pbmax + 1], order m stored at m + 2 pbmax
  const cd* t_m2m;       // [n_levels][4][4 pbmax + 1]
  const cd* t_l2l;       // [n_levels][4][4 pbmax + 1]
  cd* mpole;
  cd* local;
  cd* lpq;               // [n_coef] leaf cos/sin coefficients of L2P (see unscale_leaf_locals_kernel)
  const int* ffs;        // [n_levels] power-of-two scale exponent of the float-float kernels
  float2* loc32;         // [n_coef] leaf locals gamma_n 2^{ffs |n|} (mixed L2QBXL)
  const double *conv, *iconv;  // [n_levels][pbmax + 1] s^j / sig_j and its inverse (mixed path)
  const double* lsig;    // [n_levels][pbmax + 1] log sig_j
  const double* isig;    // [n_levels][pbmax + 2] 1 / sig_min(j, pb) (mixed P2M)
  const float2* isf;     // the same times 2^{ffs j}, float-float
  const double2* sigr;   // [n_levels][pbmax + 2] (sig_{j-1} / sig_j, sig_{j+1} / sig_j)
  double k, ik, side;    // wavenumber, 1 / k, root box side
  FfUnits U;             // units of the float-float kernels
  int pbmax, p, n_levels, has_S, has_D;
};

__device__ __forceinline__ const double* pw_row(const Fmm& F, int l) { return F.pw + (size_t)l * (2 * F.pbmax + 3); }
// e: every FP64 result of the mixed path is multiplied by 2^e
__device__ __forceinline__ int out_exp(const Fmm& F) { return __ldg(F.sexp); }
__device__ __forceinline__ const double* ipw_row(const Fmm& F, int l) { return F.ipw + (size_t)l * (F.pbmax + 2); }

// Unnormalised Miller recurrence for J_0..J_M of x into row[0..M]; returns the
// normalisation (divide by it). Rescales the stored part when values grow.
__device__ double miller_row(double x, int M, double* row, int stride) {
  if (x < 1e-8) {
    double t = 1.0;
    for (int i = 0; i <= M; ++i) {
      row[i * stride] = t;
      t *= 0.5 * x / (double)(i + 1);
    }
    return 1.0;
  }
  const double inv = 2.0 / x;
  const int N = miller_start(M, x);  // > M + 1: every row entry is written
  double fn1 = 0.0, fn = 0x1p-600, sum = 0.0, dn = (double)N;
  for (int n = N; n >= 1; --n) {
    const double fm = fma(dn * inv, fn, -fn1);  // f_{n-1} = (2n/x) f_n - f_{n+1}
    dn -= 1.0;
    if ((n & 1) == 0) sum += fn;
    if (n - 1 <= M) row[(n - 1) * stride] = fm;
    fn1 = fn;
    fn = fm;
    // rescale by 2^-332 (exact) once |f| reaches 2^332: an integer test on the
    // exponent field
    if ((__double2hiint(fn) & 0x7FFFFFFF) >= (1355 << 20)) {
      const double sc = 0x1p-332;
      fn *= sc;
      fn1 *= sc;
      sum *= sc;
      for (int i = n - 1; i <= M; ++i) row[i * stride] *= sc;
    }
  }
  return fn + 2.0 * sum;
}

// ---------------------------------------------------------------- translation tables
// One thread per (level, item): items 0..48 M2L offset classes, 49..52 M2M
// quadrants, 53..56 L2L quadrants. Rows have stride 4 pbmax + 1 with order m
// at m + 2 pbmax; only the orders a level's translations read are written:
// |m| <= 2 pb_l for M2L, |m| <= pb_l + pb_{l+1} for M2M / L2L. Levels 0 and 1
// carry no expansions.
__global__ void tables_kernel(int n_levels, double side, double k, int pbmax,
                              const int* __restrict__ lpb, const double* __restrict__ scale,
                              cd* __restrict__ t_m2l, cd* __restrict__ t_m2m,
                              cd* __restrict__ t_l2l, double* __restrict__ jwork) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n_levels * 57) return;
  const int l = g / 57, item = g % 57;
  const int TS = 4 * pbmax + 1, C = 2 * pbmax;
  const int pb = lpb[l];
  if (l < 2 || pb == 0) return;
  const double sl = side / (double)(1 << l);
  if (item < 49) {
    cd* out = t_m2l + ((size_t)l * 49 + item) * TS + C;
    const int dx = item / 7 - 3, dy = item % 7 - 3;  // (ix_b - ix_c, iy_b - iy_c)
    if (max(abs(dx), abs(dy)) < 2) return;          // not a V-list offset
    const int M = 2 * pb;
    const double s = scale[l];
    const double Dx = dx * sl, Dy = dy * sl, r = sqrt(Dx * Dx + Dy * Dy), x = k * r;
    const cd e1 = mk(Dx / r, Dy / r);
    cd h0, h1;
    hankel01(x, h0, h1);
    cd hm1 = h0, hm = cscale(h1, s);  // scaled H_m s^m
    cd e = mk(1.0, 0.0);
    out[0] = h0;
    for (int m = 1; m <= M; ++m) {
      e = cmul(e, e1);
      out[m] = cmul(hm, e);
      const double sg = (m & 1) ? -1.0 : 1.0;
      out[-m] = cscale(cmul(hm, cconj(e)), sg);
      // next: H_{m+1} s^{m+1} = (2m/x) s H_m s^m - s^2 H_{m-1} s^{m-1}
      const cd hn = csub(cscale(hm, 2.0 * m * s / x), cscale(hm1, s * s));
      hm1 = hm;
      hm = hn;
    }
    return;
  }
  if (l + 1 >= n_levels) return;
  const bool m2m = item < 53;
  const int c = m2m ? item - 49 : item - 53;
  cd* out = (m2m ? t_m2m : t_l2l) + ((size_t)l * 4 + c) * TS + C;
  const int M = pb + lpb[l + 1];
  // child centre minus parent centre, child side = sl/2
  const double cs = 0.5 * sl;
  const double dx = ((c & 1) - 0.5) * cs, dy = ((c >> 1) - 0.5) * cs;
  const double r = sqrt(dx * dx + dy * dy), x = k * r;
  double* J = jwork + (size_t)g * (2 * pbmax + 1);
  const double norm = miller_row(x, M, J, 1);
  const cd e1 = mk(dx / r, dy / r);
  cd e = mk(1.0, 0.0);
  for (int m = 0; m <= M; ++m) {
    const double j = J[m] / norm;
    const double sg = (m & 1) ? -1.0 : 1.0;
    if (m2m) {  // conj(V_m) = J_m e^{-im th}; conj(V_{-m}) = (-1)^m J_m e^{im th}
      out[m] = cscale(cconj(e), j);
      out[-m] = cscale(e, sg * j);
    } else {    // (-1)^m V_m = (-1)^m J_m e^{im th}; (-1)^m V_{-m} = J_m e^{-im th}
      out[m] = cscale(e, sg * j);
      out[-m] = cscale(cconj(e), j);
    }
    e = cmul(e, e1);
  }
}

// Per level: pw[j] = s^j for j <= 2 pb_l + 2, ipw[j] = s^-j for j <= pb_l + 1 (rest 0).
__global__ void powers_kernel(int n_levels, int pbmax, const int* __restrict__ lpb,
                              const double* __restrict__ scale, double* __restrict__ pw,
                              double* __restrict__ ipw) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= n_levels) return;
  const double s = scale[l];
  const int pb = lpb[l];
  double a = 1.0;
  for (int j = 0; j < 2 * pbmax + 3; ++j) {
    pw[(size_t)l * (2 * pbmax + 3) + j] = j <= 2 * pb + 2 ? a : 0.0;
    a *= s;
  }
  a = 1.0;
  for (int j = 0; j < pbmax + 2; ++j) {
    ipw[(size_t)l * (pbmax + 2) + j] = j <= pb + 1 ? a : 0.0;
    if (j <= pb + 1) a /= s;
  }
}

// ---------------------------------------------------------------- strengths
// Sorted strengths; for the mixed path (str_exp set) times 2^-e, e the exponent of the
// largest of them, so that a density of any size keeps the FP32 stages in range
// (out_exp: 2^e is put back where FP64 results are formed; every step is the same to
// the bit for 2^n times a density), and their FP32 forms, with the dipole factors
// A = d (k/2) nu and B = d (k/2) conj(nu) (nu = n_x + i n_y) formed once per source
// instead of once per (source, centre) pair.
__global__ void gather_strengths_kernel(int64_t n, const int* __restrict__ perm,
                                        const cd* __restrict__ q, const cd* __restrict__ d,
                                        const double2* __restrict__ snrm, double k,
                                        cd* __restrict__ qs, cd* __restrict__ ds,
                                        float2* __restrict__ q32, float4* __restrict__ ab32,
                                        float4* __restrict__ dn32, float4* __restrict__ qf,
                                        float4* __restrict__ df, float4* __restrict__ nf,
                                        const int* __restrict__ str_exp, int n_exp,
                                        int* __restrict__ sexp) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int at = i < n ? perm[i] : 0;
  cd qi = q[at], di = d[at];
  if (str_exp) {
    int e = 0;
    for (int j = threadIdx.x; j < n_exp; j += 256) e = max(e, str_exp[j]);
    e = block_exponent(e);
    e = e == 0 ? 0 : min(e - 1023, 1022);  // 2^e and 2^-e are normal
    if (i == 0) *sexp = e;
    qi = cscale(qi, pow2d(-e));
    di = cscale(di, pow2d(-e));
  }
  if (i >= n) return;
  qs[i] = qi;
  ds[i] = di;
  if (q32) {
    const cd dk = cscale(di, 0.5 * k);
    const cd nu = mk(snrm[i].x, snrm[i].y);
    const cd A = cmul(dk, nu), B = cmul(dk, cconj(nu));
    q32[i] = make_float2((float)qi.x, (float)qi.y);
    ab32[i] = make_float4((float)A.x, (float)A.y, (float)B.x, (float)B.y);
    dn32[i] = make_float4((float)dk.x, (float)dk.y, (float)nu.x, (float)nu.y);
    auto two = [](cd v) {
      const ff a = ff_round(v.x), b = ff_round(v.y);
      return make_float4(a.h, a.l, b.h, b.l);
    };
    qf[i] = two(qi);
    df[i] = two(cscale(di, k));
    nf[i] = two(nu);
  }
}

// ---------------------------------------------------------------- P2M (Stage 2)
// Shared memory of the source-row kernels (P2M, P2L): an accumulator per output
// order, then up to kChunk rows of 2 pb + 3 table values and three strengths.
__host__ __device__ inline size_t rows_smem(int pb, int chunk) {
  return ((size_t)(2 * pb + 1) + (size_t)chunk * (2 * pb + 6)) * sizeof(cd);
}
__host__ __device__ inline int rows_chunk(int pb, size_t sm_bytes) {
  const size_t per = (size_t)(2 * pb + 6) * sizeof(cd);
  const size_t avail = sm_bytes - (size_t)(2 * pb + 1) * sizeof(cd);
  const size_t c = avail / per;
  return (int)(c < (size_t)kChunk ? c : (size_t)kChunk);
}

// Row of source i for the multipole of a box with centre m, order pb and
// scale s: row[t] = conj(V_t(y_i - m)) / s^|t|, |t| <= pb + 1 (row points at
// t = 0), and the source's charge and dipole factors in sq, sa, sb.
__device__ __forceinline__ void p2m_fill_row(const Fmm& F, int i, double2 m, double is, int pb,
                                             cd* row, cd& sq, cd& sa, cd& sb) {
  const double dx = F.sxy[i].x - m.x, dy = F.sxy[i].y - m.y;
  const double rr = sqrt(dx * dx + dy * dy);
  // J_0..J_{pb+1} (unnormalised) into the real parts of row[0..pb+1]
  const double norm = miller_row(F.k * rr, pb + 1, (double*)row, 2);
  const cd em = rr > 0.0 ? mk(dx / rr, -dy / rr) : mk(1.0, 0.0);  // e^{-i th}
  cd e = mk(1.0, 0.0);
  double f = 1.0 / norm;
  for (int j = 0; j <= pb + 1; ++j) {
    const double v = row[j].x * f;                // J_j / s^j
    const cd c = cscale(e, v);                    // conj(V_j) / s^j
    row[j] = c;
    if (j > 0) row[-j] = (j & 1) ? mk(-c.x, c.y) : mk(c.x, -c.y);  // (-1)^j conj(c)
    e = cmul(e, em);
    f *= is;
  }
  const cd dk = cscale(F.ds[i], 0.5 * F.k);
  const cd nu = mk(F.snrm[i].x, F.snrm[i].y);
  sq = F.qs[i];
  sa = cmul(dk, cconj(nu));
  sb = cmul(dk, nu);
}

// Order n of a box's multipole from rows j0..j1 of the staged rows:
// a_n = sum_j [q_j row_j[n] + s^{|n-1| - |n|} A_j row_j[n-1] - s^{|n+1| - |n|} B_j row_j[n+1]]
// (charge and dipole terms in separate sums, each scaled once).
__device__ __forceinline__ cd p2m_order(const Fmm& F, const cd* rows, int RW, const cd* sq,
                                        const cd* sa, const cd* sb, int j0, int j1, int n,
                                        double s, double is) {
  const int an = abs(n);
  // conj(V_{n-+1})/s^|n| = row[n-+1] s^{|n-+1| - |n|}
  const double fm = (abs(n - 1) > an) ? s : is;
  const double fp = (abs(n + 1) > an) ? s : is;
  cd aq = mk(0.0, 0.0), aa = mk(0.0, 0.0), ab = mk(0.0, 0.0);
  for (int j = j0; j < j1; ++j) {
    const cd* row = rows + j * RW;
    if (F.has_S) cfma(aq, sq[j], row[n]);
    if (F.has_D) {
      cfma(aa, sa[j], row[n - 1]);
      cfma(ab, sb[j], row[n + 1]);
    }
  }
  return cadd(aq, csub(cscale(aa, fm), cscale(ab, fp)));
}

// P2M work: every source leaf's sources are cut into segments of at most a
// row chunk; segments of one level are packed into items of up to a chunk of
// sources (item = (first segment, segments, first packed source, sources)),
// so small leaves share a CTA and large ones spread over several. One warp
// fills the item's rows with full lanes; then the threads run over
// (segment, order) pairs and write each segment's part of its leaf's multipole
// to partial[seg_poff[segment] + n + pb]; p2m_sum_kernel adds a leaf's
// segments in order.
__global__ void __launch_bounds__(kThreads) p2m_item_kernel(Fmm F, const int4* __restrict__ items,
                                                            const int* __restrict__ seg_leaf,
                                                            const int2* __restrict__ seg_row,
                                                            const long long* __restrict__ seg_poff,
                                                            const int* __restrict__ src,
                                                            const int* __restrict__ src_leaf,
                                                            cd* __restrict__ partial,
                                                            unsigned sm_bytes) {
  extern __shared__ cd smem[];
  const int4 it = items[blockIdx.x];
  const int l = F.level[seg_leaf[it.x]];
  const int pb = F.lpb[l], Q = 2 * pb + 1, RW = 2 * pb + 3;
  const int chunk = rows_chunk(pb, sm_bytes);  // >= it.w
  cd* rows = smem;                        // [chunk][RW]
  cd* sq = rows + chunk * RW;             // [chunk]
  cd* sa = sq + chunk;                    // [chunk]
  cd* sb = sa + chunk;                    // [chunk]
  const double s = F.scale[l], is = 1.0 / s;
  if ((int)threadIdx.x < it.w) {
    const int j = threadIdx.x;
    p2m_fill_row(F, src[it.z + j], F.centre[src_leaf[it.z + j]], is, pb, rows + j * RW + (pb + 1),
                 sq[j], sa[j], sb[j]);
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < it.y * Q; idx += kThreads) {
    const int u = idx / Q, n = idx % Q - pb;
    const int2 rr = seg_row[it.x + u];
    partial[seg_poff[it.x + u] + n + pb] =
        p2m_order(F, rows + (pb + 1), RW, sq, sa, sb, rr.x, rr.x + rr.y, n, s, is);
  }
}

// mpole(leaves[t]) = sum of its segments' partial multipoles, in order
// (segments lseg[t]..lseg[t+1]).
__global__ void __launch_bounds__(kThreads) p2m_sum_kernel(Fmm F, const int* __restrict__ leaves,
                                                           const int* __restrict__ lseg,
                                                           const long long* __restrict__ seg_poff,
                                                           const cd* __restrict__ partial) {
  const int t = blockIdx.x, b = leaves[t];
  const int Q = 2 * F.lpb[F.level[b]] + 1;
  cd* dst = F.mpole + F.eoff[b];
  for (int n = threadIdx.x; n < Q; n += kThreads) {
    cd sum = mk(0.0, 0.0);
    for (int g = lseg[t]; g < lseg[t + 1]; ++g) sum = cadd(sum, partial[seg_poff[g] + n]);
    dst[n] = sum;
  }
}

// ---------------------------------------------------------------- M2M (Stage 2), L2L (Stage 7)
// FP64. a_s = sum over the children and |n| <= pc of a'_n conj(V_{s-n}), and
// gamma'_s = sum_{|n| <= pp} gamma_n (-1)^{s-n} V_{s-n}. The four children of a box lie
// at the same distance and at the angles pi/4 + rho pi/2, so that with rotations by
// eighth turns both are a real matrix product J_{s-n}, and the rotations of the four
// children differ by quarter turns, which depend on s - n mod 4 only:
//   M2M  a_s = e^{-i s pi/4} sum_n J_{s-n} b_{(n-s) mod 4, n},
//        b_{j,n} = sum_rho i^{rho j} e^{i n pi/4} a'_{rho,n};
//   L2L  gamma'_{rho,s} = e^{i s pi/4} sum_k i^{rho k} t_k,
//        t_k = sum over n = s - k mod 4 of J_{n-s} e^{-i n pi/4} gamma_n.
// 2 FMAs per (n, s) and parent where the four complex products take 16. The matrices
// T[n][s] hold the powers of the scaled coefficients and 1/sqrt 2 for each odd order of
// the eighth turns (turn8 leaves it out).
// A CTA takes a parent; warp w sums the terms n = w mod 4 (counted from the lowest
// order) of 32 orders s, one per lane, and the warps join the four sums. The orders s
// are taken 32 at a time, gridDim.y apart. Bound by the FP64 pipe (304 FMAs per clock
// over the chip). M2M and L2L of 25 ellipses 0.73 and 0.72 ms -> 0.28 and 0.32 against
// the exact split of the four complex products on the tensor cores, which this replaces
// (its conversions to and from digits cost more than the products), of 200 ellipses
// 2.57 -> 1.48 and 1.98 -> 1.81, of the 8192-node starfish 0.19 and 0.15 -> 0.07 and
// 0.08; also the faster one at box orders of 573.
constexpr int child_at(int rho) { return (0x4B >> (2 * rho)) & 3; }  // quadrant at pi/4 + rho pi/2
__device__ __forceinline__ cd turn4(cd v, int q) {  // i^q v
  if (q & 1) v = mk(-v.y, v.x);
  if (q & 2) v = mk(-v.x, -v.y);
  return v;
}
__device__ __forceinline__ cd turn8(cd v, int m) {  // e^{i m pi/4} v, sqrt 2 times for odd m
  if (m & 1) v = mk(v.x - v.y, v.x + v.y);
  return turn4(v, m >> 1);
}
__device__ __forceinline__ void dft4(cd (&v)[4]) {  // v_j <- sum_rho i^{rho j} v_rho
  const cd a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
  const cd c = cadd(v[1], v[3]), d = mk(v[3].y - v[1].y, v[1].x - v[3].x);
  v[0] = cadd(a, c);
  v[2] = csub(a, c);
  v[1] = cadd(b, d);
  v[3] = csub(b, d);
}
// The matrix of parent level l: M2M from child order n to parent order s, L2L from
// parent to child; from the tables of the quadrant at pi/4. Grid: n, threads over s.
template <bool M2M>
__global__ void fold64_matrix_kernel(int l, int pp, int pc, int pbmax, const cd* __restrict__ table,
                                     const double* __restrict__ pw, const double* __restrict__ ipw,
                                     double* __restrict__ T) {
  const int pn = M2M ? pc : pp, ps = M2M ? pp : pc;
  const int n = (int)blockIdx.x - pn;
  const cd* v = table + ((size_t)l * 4 + child_at(0)) * (4 * pbmax + 1) + 2 * pbmax;
  const double* pwc = pw + (size_t)(l + 1) * (2 * pbmax + 3);
  const double* ipp = ipw + (size_t)l * (pbmax + 2);
  double* dst = T + (size_t)(n + pn) * (2 * ps + 1) + ps;
  for (int s = (int)threadIdx.x - ps; s <= ps; s += blockDim.x) {
    const cd e = v[s - n];  // J_{s-n} e^{-i (s-n) pi/4} (M2M), J_{n-s} e^{i (s-n) pi/4} (L2L)
    double c, sn;
    sincospi(0.25 * (M2M ? s - n : n - s), &sn, &c);
    double f = M2M ? pwc[abs(n)] * ipp[abs(s)] : pwc[abs(s)] * ipp[abs(n)];
    if ((n & 1) && (s & 1)) f *= 0.5;
    else if ((n | s) & 1) f *= 0.70710678118654752440;
    dst[s] = (e.x * c - e.y * sn) * f;
  }
}
constexpr int kFoldCols = 32;
// sum_{j < N} M[j * ld] x[j * xs]
__device__ __forceinline__ cd real_sum(const double* __restrict__ M, size_t ld, int N,
                                       const cd* __restrict__ x, int xs) {
  cd sum = mk(0.0, 0.0);
#pragma unroll 4
  for (int j = 0; j < N; ++j) {
    const double t = M[(size_t)j * ld];
    const cd v = x[(size_t)j * xs];
    sum.x = fma(t, v.x, sum.x);
    sum.y = fma(t, v.y, sum.y);
  }
  return sum;
}
__global__ void __launch_bounds__(kThreads) m2m_kernel(Fmm F, const int* __restrict__ boxes,
                                                       const double* __restrict__ T) {
  extern __shared__ cd smem[];  // [Qc][4], then [4][kFoldCols]
  const int b = boxes[blockIdx.x];
  const int l = F.level[b];
  const int pp = F.lpb[l], pc = F.lpb[l + 1];
  const int Qc = 2 * pc + 1, Qp = 2 * pp + 1;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  cd* red = smem + 4 * Qc;
  const cd* src[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int d = F.child[4 * b + child_at(c)];
    src[c] = d >= 0 ? F.mpole + F.eoff[d] : nullptr;
  }
  for (int i = threadIdx.x; i < Qc; i += kThreads) {
    cd v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = src[c] ? turn8(src[c][i], i - pc) : mk(0.0, 0.0);
    dft4(v);
#pragma unroll
    for (int j = 0; j < 4; ++j) smem[4 * i + j] = v[j];
  }
  __syncthreads();
  for (int s0 = blockIdx.y * kFoldCols; s0 < Qp; s0 += kFoldCols * gridDim.y) {
    const int at = s0 + lane, s = at - pp;
    const int j = (w - pc - s) & 3;
    cd sum = mk(0.0, 0.0);
    if (at < Qp && w < Qc)
      sum = real_sum(T + (size_t)w * Qp + at, 4 * (size_t)Qp, (Qc - w + 3) / 4, smem + 4 * w + j, 16);
    __syncthreads();
    red[w * kFoldCols + lane] = sum;
    __syncthreads();
    if (w == (s0 / kFoldCols & 3) && at < Qp) {
      cd v = cadd(cadd(red[lane], red[kFoldCols + lane]),
                  cadd(red[2 * kFoldCols + lane], red[3 * kFoldCols + lane]));
      F.mpole[F.eoff[b] + at] = turn8(v, -s);
    }
  }
}
__global__ void __launch_bounds__(kThreads) l2l_kernel(Fmm F, const int* __restrict__ boxes,
                                                       const double* __restrict__ T) {
  extern __shared__ cd smem[];  // [Qp], then [4][kFoldCols]
  const int b = boxes[blockIdx.x];
  const int l = F.level[b];
  const int pp = F.lpb[l], pc = F.lpb[l + 1];
  const int Qp = 2 * pp + 1, Qc = 2 * pc + 1;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  cd* red = smem + Qp;
  const cd* lp = F.local + F.eoff[b];
  for (int i = threadIdx.x; i < Qp; i += kThreads) smem[i] = turn8(lp[i], pp - i);
  const int d = F.child[4 * b + child_at(w)];  // warp w stores the child at rho = w
  cd* dl = d >= 0 ? F.local + F.eoff[d] : nullptr;
  __syncthreads();
  for (int s0 = blockIdx.y * kFoldCols; s0 < Qc; s0 += kFoldCols * gridDim.y) {
    const int at = s0 + lane, s = at - pc;
    cd sum = mk(0.0, 0.0);
    if (at < Qc && w < Qp)
      sum = real_sum(T + (size_t)w * Qc + at, 4 * (size_t)Qc, (Qp - w + 3) / 4, smem + w, 4);
    __syncthreads();
    red[w * kFoldCols + lane] = sum;
    __syncthreads();
    if (dl && at < Qc) {  // sum_k i^{w k} t_k, t_k in the sums of warp (s + pp - k) mod 4
      cd v = red[((s + pp) & 3) * kFoldCols + lane];
#pragma unroll
      for (int k = 1; k < 4; ++k)
        v = cadd(v, turn4(red[((s + pp - k) & 3) * kFoldCols + lane], w * k));
      dl[at] = cadd(dl[at], turn8(v, s));
    }
  }
}
size_t m2m_smem(int pc) { return (4 * (size_t)(2 * pc + 1) + 4 * kFoldCols) * sizeof(cd); }
size_t l2l_smem(int pp) { return ((size_t)(2 * pp + 1) + 4 * kFoldCols) * sizeof(cd); }
// blocks along the orders: all of a parent's orders in one where there are parents
// enough, so that they are staged once
unsigned fold_split(int nb, int Q) {
  return std::min(nblk(Q, kFoldCols), std::max(1u, 8u * 152u / (unsigned)nb));
}

// ---------------------------------------------------------------- M2L (Stage 4)
// lh_l += (-1)^l sum_n What_{n+l} mh_n c(l,n), What_m = s^|m| W_m(m_b - m_c),
// c(l,n) = s^{2 min(|l|,|n|)} when l and n have opposite signs, else 1: both
// precisions run it as tile GEMMs over dense per-(level, offset class)
// matrices (mixed.cu).

// ---------------------------------------------------------------- P2L (Stage 6)
// lh_n += s^|n| sum_j [q_j W_n + d_j (k/2)(nu_j W_{n-1} - conj(nu_j) W_{n+1})](y_j - m_b)
// over the sources of the boxes in b's X list. Work items: up to one row chunk
// of an X box's sources (its X list's leaves, concatenated in list order), so
// that a box's work spreads over several CTAs and every chunk is full. One
// warp fills a row per source with Wh_t = s^|t| W_t, |t| <= pb + 1; then all
// threads form the item's part of lh_n (the charge and the two dipole terms in
// separate sums, scaled once) into partial[poff[item] + n + pb], and
// p2l_sum_kernel adds each box's items in order.
__global__ void __launch_bounds__(kThreads) p2l_item_kernel(Fmm F, const int4* __restrict__ items,
                                                            const int* __restrict__ src,
                                                            const long long* __restrict__ poff,
                                                            cd* __restrict__ partial,
                                                            unsigned sm_bytes) {
  extern __shared__ cd smem[];
  const int4 it = items[blockIdx.x];  // (box, first position in src, sources, -)
  const int b = it.x, cnt = it.z;
  const int l = F.level[b];
  const int pb = F.lpb[l], RW = 2 * pb + 3;  // row: Wh_t, |t| <= pb+1
  const int chunk = rows_chunk(pb, sm_bytes);  // >= cnt (items are cut to fit)
  cd* rows = smem;                        // [chunk][RW]
  cd* sq = rows + chunk * RW;             // [chunk]
  cd* sa = sq + chunk;                    // [chunk]  A = d (k/2) nu
  cd* sb = sa + chunk;                    // [chunk]  B = d (k/2) conj(nu)
  const double s = F.scale[l], is = 1.0 / s;
  const double2 m = F.centre[b];
  const double hk = 0.5 * F.k;
  if ((int)threadIdx.x < cnt) {
    const int i = src[it.y + threadIdx.x];
    const double dx = F.sxy[i].x - m.x, dy = F.sxy[i].y - m.y;
    const double rr = sqrt(dx * dx + dy * dy), irr = 1.0 / rr;
    const double x = F.k * rr, ix = 1.0 / x;
    const cd e1 = mk(dx * irr, dy * irr);
    cd h0, h1;
    hankel01(x, ix, h0, h1);
    const double c1 = 2.0 * s * ix, s2 = s * s;  // Wh_{j+1} = j c1 Wh_j - s2 Wh_{j-1}
    cd* row = rows + threadIdx.x * RW + (pb + 1);   // row[t], t = -(pb+1)..pb+1
    cd hm1 = h0, hm = cscale(h1, s), ee = mk(1.0, 0.0);
    row[0] = h0;
    for (int j = 1; j <= pb + 1; ++j) {
      ee = cmul(ee, e1);
      const double ac = hm.x * ee.x, bd = hm.y * ee.y, ad = hm.x * ee.y, bc = hm.y * ee.x;
      row[j] = mk(ac - bd, ad + bc);                                       // s^j W_j
      row[-j] = (j & 1) ? mk(-(ac + bd), ad - bc) : mk(ac + bd, bc - ad);  // s^j W_{-j}
      const cd hn = csub(cscale(hm, j * c1), cscale(hm1, s2));
      hm1 = hm;
      hm = hn;
    }
    const cd dk = cscale(F.ds[i], hk);
    const cd nu = mk(F.snrm[i].x, F.snrm[i].y);
    sq[threadIdx.x] = F.qs[i];
    sa[threadIdx.x] = cmul(dk, nu);
    sb[threadIdx.x] = cmul(dk, cconj(nu));
  }
  __syncthreads();
  cd* dst = partial + poff[blockIdx.x] + pb;
  for (int n = (int)threadIdx.x - pb; n <= pb; n += kThreads) {
    const int an = abs(n);
    // s^|n| W_{n-1} = Wh_{n-1} s^{|n| - |n-1|}, s^|n| W_{n+1} = Wh_{n+1} s^{|n| - |n+1|}
    const double fm = (abs(n - 1) > an) ? is : s;
    const double fp = (abs(n + 1) > an) ? is : s;
    cd aq = mk(0.0, 0.0), aa = mk(0.0, 0.0), ab = mk(0.0, 0.0);
    for (int j = 0; j < cnt; ++j) {
      const cd* row = rows + j * RW + (pb + 1);
      if (F.has_S) cfma(aq, sq[j], row[n]);
      if (F.has_D) {
        cfma(aa, sa[j], row[n - 1]);
        cfma(ab, sb[j], row[n + 1]);
      }
    }
    dst[n] = cadd(aq, csub(cscale(aa, fm), cscale(ab, fp)));
  }
}

// lh(xbox[t]) += its items' partial coefficients, in item order.
__global__ void __launch_bounds__(kThreads) p2l_sum_kernel(Fmm F, const int* __restrict__ xbox,
                                                           const int* __restrict__ boff,
                                                           const long long* __restrict__ poff,
                                                           const cd* __restrict__ partial) {
  const int t = blockIdx.x, b = xbox[t];
  const int pb = F.lpb[F.level[b]], Q = 2 * pb + 1;
  cd* dst = F.local + F.eoff[b];
  for (int n = threadIdx.x; n < Q; n += kThreads) {
    cd sum = mk(0.0, 0.0);
    for (int it = boff[t]; it < boff[t + 1]; ++it) sum = cadd(sum, partial[poff[it] + n]);
    dst[n] = cadd(dst[n], sum);
  }
}

// ---------------------------------------------------------------- targets (Stages 3, 5, 8)
// CTA per leaf; one thread per target of the leaf (strided). Only targets that
// are not associated with a QBX centre are evaluated.
// L2P writes out[t], M2P and P2P add to it.
// Sources of a list of boxes, concatenated: the boxes of leaf b's U list
// (U.idx[uoff[b]..uoff[b+1])) followed by the boxes xidx[x0..x1) (the W-list
// boxes summed directly for one centre; empty for targets). Lane `lane` takes
// the sources t = lane, lane + 32, ... of the concatenation (a cursor per lane
// walks the boxes), so a warp runs ceil(total / 32) iterations.
struct SourceCursor {
  const int* uidx;   // the U-list index array
  const int2* rsrc;  // source range of every box
  int u0, nu, x0, nx;
  const int* xidx;
  __device__ int box(int e) const { return e < nu ? uidx[u0 + e] : xidx[x0 + e - nu]; }
  __device__ int total() const {
    int t = 0;
    for (int e = 0; e < nu + nx; ++e) {
      const int2 r = rsrc[box(e)];
      t += r.y - r.x;
    }
    return t;
  }
};

template <int W = 32, typename Fn>
__device__ __forceinline__ void deal_sources(const SourceCursor& sc, int lane, Fn&& fn) {
  const int tot = sc.total();
  int e = 0, base = 0;
  int2 r = sc.nu + sc.nx > 0 ? sc.rsrc[sc.box(0)] : make_int2(0, 0);
  for (int t = lane; t < tot; t += W) {
    while (t >= base + (r.y - r.x)) {  // advance to the box holding source t
      base += r.y - r.x;
      r = sc.rsrc[sc.box(++e)];
    }
    fn(r.x + (t - base));
  }
}

// L2P: one thread per direct target (sorted index list), from the local
// coefficients of its leaf in cosine/sine form (P_m, Q_m); adds to out. The
// backward recurrence yields f_m for descending m, and Clenshaw's recurrences
// for the cosine and sine sums run in the same loop (two FMAs per real
// component and order, no complex products).
__device__ __forceinline__ cd l2p_value(const Fmm& F, int i, int b) {
  const int pb = F.lpb[F.level[b]];
  const cd* g = F.local + F.eoff[b];
  const double2 m = F.centre[b];
  const double dx = F.txy[i].x - m.x, dy = F.txy[i].y - m.y;
  const double d2 = dx * dx + dy * dy;
  const bool at_centre = (__double2hiint(d2) | __double2loint(d2)) == 0;
  const double ir = at_centre ? 0.0 : rsqrt(d2), x = F.k * (d2 * ir);
  const cd e1 = at_centre ? mk(1.0, 0.0) : mk(dx * ir, dy * ir);
  // psi = sum_m f_m [g_m e^{-im th} + (m>0) (-1)^m g_{-m} e^{im th}] / norm
  cd acc;
  double norm;
  if (x < 1e-8) {
    // J_m(x) = (x/2)^m / m! to relative O(x^2); the terms vanish after a few
    // orders (a target a rounding distance from the leaf centre still needs
    // the m = 1 term: it is O(x) of the result, not O(x^2))
    acc = mk(0.0, 0.0);
    norm = 1.0;
    double t = 1.0;
    cd e = mk(1.0, 0.0);  // e^{i m th}
    for (int mm = 0; mm <= pb && t != 0.0; ++mm) {
      acc = cadd(acc, cscale(cmul(g[pb + mm], cconj(e)), t));
      if (mm > 0) acc = cadd(acc, cscale(cmul(g[pb - mm], e), (mm & 1) ? -t : t));
      t *= 0.5 * x / (double)(mm + 1);
      e = cmul(e, e1);
    }
  } else {
    // Miller's backward recurrence for f_m ~ J_m(x) (unnormalised), fused with
    // Clenshaw's recurrences for sum_m f_m P_m cos(m th) (u: b_{m+1}, b_{m+2})
    // and sum_m f_m Q_m sin(m th) (v), both run from m = pb down:
    //   b_m = f_m c_m + 2 cos(th) b_{m+1} - b_{m+2},
    //   sum c_m cos(m th) = b_0 - cos(th) b_1,  sum_{m>=1} c_m sin(m th) = sin(th) b_1.
    const cd* pq = F.lpq + F.eoff[b];
    const double c = e1.x, c2 = 2.0 * c;
    const double inv = 2.0 / x;
    const int N = miller_start(pb, x);
    double fn1 = 0.0, fn = 0x1p-600, sum = 0.0, dn = (double)N;
    // f_{n-1} = (2n/x) f_n - f_{n+1}; the sum of the even orders normalises
    // (J_0 + 2 sum J_{2k} = 1); a power of two rescales everything kept when
    // f grows past 2^332 (an integer test on the exponent field)
    auto step = [&]() {
      const double fm = fma(dn * inv, fn, -fn1);
      fn1 = fn;
      fn = fm;
      dn -= 1.0;
    };
    int nn = N;
    for (; nn >= pb + 2; --nn) {  // orders above pb: the recurrence alone
      if ((nn & 1) == 0) sum += fn;
      step();
      if ((__double2hiint(fn) & 0x7FFFFFFF) >= (1355 << 20)) {
        fn *= 0x1p-332; fn1 *= 0x1p-332; sum *= 0x1p-332;
      }
    }
    cd u1 = mk(0.0, 0.0), u2 = u1, v1 = u1, v2 = u1;
    for (; nn >= 1; --nn) {
      if ((nn & 1) == 0) sum += fn;
      step();
      const int mm = nn - 1;  // fn = f_mm
      const cd P = pq[mm];
      const cd u0 = mk(fma(fn, P.x, fma(c2, u1.x, -u2.x)), fma(fn, P.y, fma(c2, u1.y, -u2.y)));
      u2 = u1;
      u1 = u0;
      if (mm >= 1) {
        const cd Qm = pq[pb + mm];
        const cd v0 = mk(fma(fn, Qm.x, fma(c2, v1.x, -v2.x)), fma(fn, Qm.y, fma(c2, v1.y, -v2.y)));
        v2 = v1;
        v1 = v0;
      }
      if ((__double2hiint(fn) & 0x7FFFFFFF) >= (1355 << 20)) {
        const double sc = 0x1p-332;
        fn *= sc; fn1 *= sc; sum *= sc;
        u1 = cscale(u1, sc); u2 = cscale(u2, sc); v1 = cscale(v1, sc); v2 = cscale(v2, sc);
      }
    }
    acc = mk(fma(-c, u2.x, u1.x) + e1.y * v1.x, fma(-c, u2.y, u1.y) + e1.y * v1.y);
    norm = fn + 2.0 * sum;
  }
  return cscale(acc, 1.0 / norm);
}

__global__ void __launch_bounds__(kThreads) l2p_kernel(Fmm F, const int* __restrict__ dtgt,
                                                       const int* __restrict__ tleaf, int n,
                                                       cd* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int i = dtgt[t];
  cd* dst = out + F.tid[i];
  *dst = cadd(*dst, l2p_value(F, i, tleaf[i]));
}


// The multipoles that M2P reads in cosine/sine form: at entry eoff[b] + b of pq
// (2 pb + 2 entries per box) the pairs (P_m, Q_m), m = 0..pb, of
//   a_m H_m e^{i m th} + a_{-m} H_{-m} e^{-i m th} = H_m (P_m cos m th + Q_m sin m th),
//   P_m = a_m + (-1)^m a_{-m},  Q_m = i (a_m - (-1)^m a_{-m}),  P_0 = a_0, Q_0 = 0,
// from the true coefficients a_n = mh_n s^|n| on levels whose H_pb stays in
// FP64's range (big[l] == 0), from mh_n on the others.
__global__ void __launch_bounds__(kThreads) mpole_pq_kernel(Fmm F, const int* __restrict__ boxes,
                                                            const int* __restrict__ big,
                                                            cd* __restrict__ pq) {
  const int b = boxes[blockIdx.x];
  const int l = F.level[b];
  const int pb = F.lpb[l];
  const bool sc = big[l] != 0;
  const double* pwl = pw_row(F, l);
  const cd* a = F.mpole + F.eoff[b] + pb;
  cd* dst = pq + F.eoff[b] + b;
  for (int m = threadIdx.x; m <= pb; m += kThreads) {
    const double f = sc ? 1.0 : pwl[m];
    cd g = m > 0 ? a[-m] : mk(0.0, 0.0);
    if (m & 1) g = mk(-g.x, -g.y);
    const cd d = csub(a[m], g);
    dst[2 * m] = cscale(cadd(a[m], g), f);
    dst[2 * m + 1] = m > 0 ? mk(-d.y * f, d.x * f) : mk(0.0, 0.0);
  }
}

// M2P: one thread per (direct target, W-list box of its leaf) pair, ordered by
// (leaf, box, target) so that the lanes of a warp read one box's coefficients;
// the value goes to the pair's slot in target order, and m2p_sum_kernel adds
// each target's pairs in order. Bound by the FP64 pipe: 15 instructions per
// order (the angular turn 4, P cos + Q sin 4, the product 4, the unscaled
// recurrence 3) against 27 with W_m and W_{-m} formed apart (25 ellipses, FP64:
// 0.67 -> 0.48 ms).
__global__ void __launch_bounds__(kThreads) m2p_pair_kernel(Fmm F, const int* __restrict__ pt,
                                                            const int* __restrict__ pbx,
                                                            const int* __restrict__ slot, int n,
                                                            const int* __restrict__ big,
                                                            const cd* __restrict__ pq,
                                                            cd* __restrict__ partial) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int i = pt[t], c = pbx[t];
  const int lc = F.level[c];
  const int pb = F.lpb[lc];
  const cd* a = pq + F.eoff[c] + c;
  const double2 mc = F.centre[c];
  const double dx = F.txy[i].x - mc.x, dy = F.txy[i].y - mc.y;
  // one reciprocal square root gives r, 1/r and 1/x: no division
  const double d2 = dx * dx + dy * dy;
  const double ir = rsqrt(d2), x = F.k * (d2 * ir), ix = ir * F.ik;
  const double co1 = dx * ir, si1 = dy * ir;
  cd h0, h1;
  hankel01(x, ix, h0, h1);
  cd sum = cmul(a[0], h0);
  double co = co1, si = si1;
  auto add = [&](int m, cd h) {
    const cd P = a[2 * m], Q = a[2 * m + 1];
    cfma(sum, mk(fma(P.x, co, Q.x * si), fma(P.y, co, Q.y * si)), h);
    const double u = fma(co, co1, -si * si1);
    si = fma(co, si1, si * co1);
    co = u;
  };
  if (!big[lc]) {  // H_{m+1} = (2m/x) H_m - H_{m-1}
    const double c2 = 2.0 * ix;
    double dm = 0.0;
    cd hp = h0, hc = h1;
    for (int m = 1; m <= pb; ++m) {
      add(m, hc);
      dm += 1.0;
      const double cm = dm * c2;
      const cd hn = mk(fma(cm, hc.x, -hp.x), fma(cm, hc.y, -hp.y));
      hp = hc;
      hc = hn;
    }
  } else {  // Wh_m = s^m H_m: Wh_{m+1} = m c1 Wh_m - s^2 Wh_{m-1}, c1 = 2 s / x
    const double s = F.scale[lc], c1 = 2.0 * s * ix, s2 = s * s;
    double dm = 0.0;
    cd hp = h0, hc = cscale(h1, s);
    for (int m = 1; m <= pb; ++m) {
      add(m, hc);
      dm += 1.0;
      const double cm = dm * c1;
      const cd hn = mk(fma(cm, hc.x, -s2 * hp.x), fma(cm, hc.y, -s2 * hp.y));
      hp = hc;
      hc = hn;
    }
  }
  partial[slot[t]] = sum;
}

// out[target] += sum of its M2P pairs, in pair order (targets wtgt[0..n)).
__global__ void m2p_sum_kernel(int n, const int* __restrict__ wtgt, const int* __restrict__ off,
                               const cd* __restrict__ partial, const int* __restrict__ tid,
                               cd* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  cd sum = mk(0.0, 0.0);
  for (int e = off[t]; e < off[t + 1]; ++e) sum = cadd(sum, partial[e]);
  cd* dst = out + tid[wtgt[t]];
  *dst = cadd(*dst, sum);
}

// P2P over the U list: one warp per direct target whose leaf's U list holds
// sources; lanes deal the sources round-robin, a shuffle tree adds them.
template <bool HS, bool HD>
__global__ void __launch_bounds__(kThreads) p2p_warp_kernel(Fmm F, const int* __restrict__ utgt,
                                                            const int* __restrict__ tleaf, int n,
                                                            cd* __restrict__ out) {
  const int t = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (t >= n) return;
  const int i = utgt[t];
  const int b = tleaf[i];
  const double k = F.k, ik = F.ik;
  const double tx = F.txy[i].x, ty = F.txy[i].y;
  cd acc = mk(0.0, 0.0);
  const SourceCursor sc{F.uidx, F.rsrc, F.uoff[b], F.uoff[b + 1] - F.uoff[b], 0, 0, nullptr};
  deal_sources(sc, lane, [&](int j) {
    const double dx = tx - F.sxy[j].x, dy = ty - F.sxy[j].y;
    const double r2 = dx * dx + dy * dy;
    if (r2 == 0.0) return;
    const double ir = rsqrt(r2), x = k * r2 * ir;
    cd h0, h1;
    hankel01_any<false, HS, HD>(x, ik * ir, h0, h1);
    if (HS) cfma(acc, F.qs[j], h0);
    if (HD) {
      const double2 nv = F.snrm[j];
      cfma(acc, F.ds[j], cscale(h1, k * (nv.x * dx + nv.y * dy) * ir));
    }
  });
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
    acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
  }
  if (lane == 0) {
    cd* dst = out + F.tid[i];
    *dst = cadd(*dst, acc);
  }
}

// ---------------------------------------------------------------- centres (Stages 3, 5, 8 "New")
// L2QBXL: alpha_s += sum_n gamma_n (-1)^{s-n} V_{s-n}(z - m_b), |s| <= p, from
// the true local coefficients gamma of the centre's leaf (leaf locals are
// unscaled in place once the downward pass is complete). A warp takes G
// centres. First each of G lanes fills its centre's row V_m = J_m(k r) e^{i m th},
// 0 <= m <= M = pb + p, in shared memory (one backward recurrence per centre);
// then the lanes take the warp's (centre, output order s) pairs and form
// alpha_s = sum_n gamma_n t_{s-n} over ascending n, with t_m = (-1)^m V_m for
// m >= 0 and t_m = (-1)^m V_m = conj(V_{-m}) for m < 0 (signs set on the bits,
// off the FP64 pipe). The result does not depend on G or on the launch.
__global__ void __launch_bounds__(32) l2qbxl_kernel(Fmm F, const int* __restrict__ cleaf,
                                                    const int* __restrict__ clist, int n_ctr,
                                                    int G, int TW, cd* __restrict__ alpha) {
  extern __shared__ cd trow[];  // [G][TW], TW > max M
  const int lane = threadIdx.x;
  const int c0 = blockIdx.x * G;
  const int p = F.p, P = 2 * p + 1;
  if (lane < G && c0 + lane < n_ctr) {
    const int i = clist[c0 + lane];
    const int b = cleaf[i];
    const int M = F.lpb[F.level[b]] + p;
    const double2 mb = F.centre[b];
    const double dx = F.cxy[i].x - mb.x, dy = F.cxy[i].y - mb.y;
    const double rr = sqrt(dx * dx + dy * dy);
    cd* row = trow + (size_t)lane * TW;
    // J_0..J_M (unnormalised) into the real parts of row[0..M]
    const double in = 1.0 / miller_row(F.k * rr, M, (double*)row, 2);
    const cd e1 = rr > 0.0 ? mk(dx / rr, dy / rr) : mk(1.0, 0.0);
    cd e = mk(1.0, 0.0);
    for (int m = 0; m <= M; ++m) {
      row[m] = cscale(e, row[m].x * in);
      e = cmul(e, e1);
    }
  }
  __syncwarp();
  constexpr unsigned long long kSign = 0x8000000000000000ull;
  const int nG = min(G, n_ctr - c0);
  for (int o = lane; o < nG * P; o += 32) {
    const int u = o / P, so = o % P - p;
    const int i = clist[c0 + u];
    const int b = cleaf[i];
    const int pb = F.lpb[F.level[b]];
    const cd* row = trow + (size_t)u * TW;
    const cd* g = F.local + F.eoff[b] + pb;
    cd a = mk(0.0, 0.0);
    for (int n = -pb; n <= pb; ++n) {
      const int m = so - n;
      const cd v = row[abs(m)];
      const unsigned long long fx = (m >= 0 && (m & 1)) ? kSign : 0ull;
      const unsigned long long fy = (m < 0) ? kSign : fx;
      const cd t = mk(__longlong_as_double(__double_as_longlong(v.x) ^ fx),
                      __longlong_as_double(__double_as_longlong(v.y) ^ fy));
      cfma(a, g[n], t);
    }
    cd* dst = alpha + (size_t)F.cid[i] * P + p + so;
    *dst = cadd(*dst, a);
  }
}


// Leaf local coefficients lh_n = gamma_n s^|n| -> gamma_n, in place, once the
// downward pass (M2L, P2L, L2L) is complete; L2P and L2QBXL read gamma. The
// same pass writes the leaf's L2P coefficients in cosine/sine form: with
// s_m = (-1)^m, the term of order m of the local expansion at (r, th) is
//   J_m(k r) [gamma_m e^{-i m th} + s_m gamma_{-m} e^{i m th}]
//     = J_m(k r) [P_m cos(m th) + Q_m sin(m th)],
//   P_m = gamma_m + s_m gamma_{-m},  Q_m = i (s_m gamma_{-m} - gamma_m),  P_0 = gamma_0,
// stored as lpq[eoff + m] = P_m (m = 0..pb), lpq[eoff + pb + m] = Q_m (m = 1..pb).
// With ff32 set (mixed path), leaves on float-float levels (ffs[l] = s) get
// 2^{s m} P_m and 2^{s m} Q_m as float4 (re h, re l, im h, im l) in the same
// places, for l2p_mixed_kernel, and 2^{s |n|} gamma_n in FP32 in loc32, for
// l2qbxl_ff_kernel.
// A CTA takes kBoxGroup leaves (see BoxGroup): bound by the FP64 pipe, whose warps
// one leaf's pb + 1 orders would not fill (L2L with this of 200 ellipses 0.51 -> 0.46 ms).
__global__ void __launch_bounds__(kThreads) unscale_leaf_locals_kernel(Fmm F,
                                                                       const int* __restrict__ leaves,
                                                                       int n_leaves, bool ff32) {
  __shared__ BoxGroup g;
  g.fill(leaves, n_leaves, F.level, F.lpb);
  for (int idx = threadIdx.x, u = 0; idx < g.start[kBoxGroup]; idx += kThreads) {
    while (idx >= g.start[u + 1]) ++u;
    const int b = g.box[u], m = idx - g.start[u], pb = g.start[u + 1] - g.start[u] - 1;
    const int l = F.level[b];
    const double ip = ipw_row(F, l)[m];
    cd* lp = F.local + F.eoff[b] + pb;
    cd* pq = F.lpq + F.eoff[b];
    float2* g32 = F.loc32 + F.eoff[b] + pb;
    const int s = ff32 ? F.ffs[l] : kNoFf;
    auto put = [&](int at, cd v) {
      if (s == kNoFf) {
        pq[at] = v;
        return;
      }
      const ff x = ff_from_f64_nan(v.x, 896 - s * m), y = ff_from_f64_nan(v.y, 896 - s * m);
      reinterpret_cast<float4*>(pq)[at] = make_float4(x.h, x.l, y.h, y.l);
    };
    auto put32 = [&](int n, cd v) {
      if (s != kNoFf)
        g32[n] = make_float2(f32_from_f64_sh(v.x, s * m), f32_from_f64_sh(v.y, s * m));
    };
    const cd gp = cscale(lp[m], ip);
    lp[m] = gp;
    put32(m, gp);
    if (m == 0) {
      put(0, gp);
      continue;
    }
    const cd gn = cscale(lp[-m], ip);
    lp[-m] = gn;
    put32(-m, gn);
    const cd sg = (m & 1) ? mk(-gn.x, -gn.y) : gn;
    put(m, cadd(gp, sg));
    const cd d = csub(sg, gp);
    put(pb + m, mk(-d.y, d.x));
  }
}


// M2QBXL: alpha_l += (-1)^l sum_n mh_n Wh_{n+l} s^{|n| - |n+l|},  Wh_m = s^|m| W_m(z - m_c),
// for the (centre, W-list box) pairs whose box is far enough from the centre's
// disk for the multipole series to converge on it ((R_c + r_z) <= kW |z - m_c|;
// the others are summed source by source with the U list in P2QBXL). Each pair
// is split over ceil((2p+1) / kM2qbxlOrders) threads, each with kM2qbxlOrders
// consecutive output orders; each writes its orders of partial[pair][2p+1],
// and m2qbxl_sum_kernel adds each centre's pairs in order. Threads walk
// m = |n + l| upwards with the Hankel recurrence; once m > p every term of
// output l has the same power factor (s^-l for n + l = m, s^l for n + l = -m),
// so those terms go to two plain sums scaled once at the end. One warp per
// block spreads the pairs over all SMs (the FP64 pipe is per SM).
constexpr int kM2qbxlOrders = 4;
constexpr int kM2qbxlBlock = 32;
// shared memory of the L2QBXL rows of one warp. FP64: 16 centres per warp at
// order 16 on 41-order leaves (the dot products keep the FP64 pipe busy);
// mixed: small enough for a dozen or more warps per SM, which hide the latency
// of the split coefficients' loads (8 centres per warp: L2QBXL 1.29 -> 1.02
// ms on ellipses-200; 4 was slower again)
constexpr size_t kL2qbxlSmem = 24 * 1024, kL2qbxlMixedSmem = 12 * 1024;
// shared memory of the split rows of one mixed-precision M2QBXL warp, and the
// pairs per warp: at most 8, so that a dozen or more warps share an SM (8 on
// ellipses-200: M2QBXL 1.08 -> 0.69 ms against 32)
constexpr size_t kM2qbxlMixedSmem = 48 * 1024;
constexpr int kM2qbxlMixedPairs = 8;
template <int PM, bool HS, bool HD>
__global__ void __launch_bounds__(kThreads) m2qbxl_pair_kernel(Fmm F, const int* __restrict__ pair_ctr,
                                                               const int* __restrict__ pair_box,
                                                               int n_pairs, cd* __restrict__ partial) {
  constexpr int LC = kM2qbxlOrders;
  const int p = F.p, P = 2 * p + 1;
  const int nparts = (P + LC - 1) / LC;
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  const int t = g / nparts, part = g % nparts;
  if (t >= n_pairs) return;
  const int i = pair_ctr[t], c = pair_box[t];
  const int lo0 = -p + part * LC;  // first output order of this thread (<= p)
  const double k = F.k;
  const int lc = F.level[c];
  const double s = F.scale[lc];
  const int pb = F.lpb[lc], M = pb + p;
  const cd* a = F.mpole + F.eoff[c];
  const double* pwl = pw_row(F, lc);
  const double* ipl = ipw_row(F, lc);
  const double2 z = F.cxy[i];
  const double2 mc = F.centre[c];
  const double dx = z.x - mc.x, dy = z.y - mc.y;
  const double rr = sqrt(dx * dx + dy * dy);
  const double x = k * rr, ix = 1.0 / x;
  const cd e1 = mk(dx / rr, dy / rr);
  cd h0, h1;
  hankel01(x, ix, h0, h1);
  const double c1 = 2.0 * s * ix, s2 = s * s;  // Wh_{m+1} = m c1 Wh_m - s2 Wh_{m-1}
  cd acc[LC], accp[LC], accq[LC];
#pragma unroll
  for (int j = 0; j < LC; ++j) acc[j] = accp[j] = accq[j] = mk(0.0, 0.0);
  cd hm1 = h0, hm = h0, ee = mk(1.0, 0.0);
  for (int mm = 0; mm <= M; ++mm) {
    if (mm == 1) { hm1 = h0; hm = cscale(h1, s); }
    if (mm >= 1) ee = cmul(ee, e1);
    // Wh_m = hm ee and Wh_{-m} = (-1)^m hm conj(ee) from the same four products
    const double ac = hm.x * ee.x, bd = hm.y * ee.y, ad = hm.x * ee.y, bc = hm.y * ee.x;
    const cd wp = mk(ac - bd, ad + bc);
    const double sm = (mm & 1) ? -1.0 : 1.0;
    const cd wq = mk(sm * (ac + bd), sm * (bc - ad));
    if (mm <= p) {  // |n| - |n + l| depends on n: per-term factors
#pragma unroll
      for (int j = 0; j < LC; ++j) {
        const int lo = lo0 + j;
        const int n1 = mm - lo;  // n + l = m
        if (lo <= p && n1 >= -pb && n1 <= pb) {
          const int ex = abs(n1) - mm;
          cfma(acc[j], cscale(a[n1 + pb], ex >= 0 ? pwl[ex] : ipl[-ex]), wp);
        }
        const int n2 = -mm - lo;  // n + l = -m
        if (mm > 0 && lo <= p && n2 >= -pb && n2 <= pb) {
          const int ex = abs(n2) - mm;
          cfma(acc[j], cscale(a[n2 + pb], ex >= 0 ? pwl[ex] : ipl[-ex]), wq);
        }
      }
    } else {  // n + l = m > 0 has n > 0, n + l = -m has n < 0: factors s^-l, s^l
#pragma unroll
      for (int j = 0; j < LC; ++j) {
        const int lo = lo0 + j;
        const int n1 = mm - lo, n2 = -mm - lo;
        const cd av = (n1 >= -pb && n1 <= pb) ? a[n1 + pb] : mk(0.0, 0.0);
        const cd aq = (n2 >= -pb && n2 <= pb) ? a[n2 + pb] : mk(0.0, 0.0);
        cfma(accp[j], av, wp);
        cfma(accq[j], aq, wq);
      }
    }
    if (mm >= 1) {
      const cd hn = csub(cscale(hm, mm * c1), cscale(hm1, s2));
      hm1 = hm;
      hm = hn;
    }
  }
  cd* dst = partial + (size_t)t * P;
#pragma unroll
  for (int j = 0; j < LC; ++j) {
    const int lo = lo0 + j;
    if (lo > p) break;
    const double fp = lo <= 0 ? pwl[-lo] : ipl[lo];  // s^-l
    const double fq = lo >= 0 ? pwl[lo] : ipl[-lo];  // s^l
    cd v = cadd(acc[j], cadd(cscale(accp[j], fp), cscale(accq[j], fq)));
    if (lo & 1) v = mk(-v.x, -v.y);
    dst[lo + p] = v;
  }
}

// alpha[centre] += sum of its pairs' partial coefficients, in pair order
// (centres clist[0..n), pairs of position t at cpo[t]..cpo[t+1]).
__global__ void m2qbxl_sum_kernel(int n, int P, const int* __restrict__ cpo,
                                  const cd* __restrict__ partial, const int* __restrict__ cid,
                                  const int* __restrict__ clist, const int* __restrict__ sexp,
                                  cd* __restrict__ alpha) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= (int64_t)n * P) return;
  const int t = (int)(g / P), l = (int)(g % P);
  const int t0 = cpo[t], t1 = cpo[t + 1];
  if (t1 == t0) return;
  cd sum = mk(0.0, 0.0);
  for (int e = t0; e < t1; ++e) sum = cadd(sum, partial[(size_t)e * P + l]);
  if (sexp) sum = cscale2(sum, *sexp);  // mixed path (out_exp)
  cd* dst = alpha + (size_t)cid[clist[t]] * P + l;
  *dst = cadd(*dst, sum);
}

// ---------------------------------------------------------------- mixed precision P2QBXL
// H_0, H_1 and the Hankel recurrence in float-float (ff.cuh); the terms are
// rounded to FP32, multiplied by the FP32 strengths and added with Kahan
// compensation; the lanes' sums are added in float-float and unscaled in FP64.
// With the recurrence in FP64 the kernel was bound by the FP64 pipe (82 % of
// its rate, 95 FP64 instructions per pair); now two FP64 subtractions per pair
// are left and FP32 issue bounds it: 104 459 centres of 200 ellipses, p = 16, 5.83
// -> 1.24 ms with what p2qbxl_pair_mixed and the half warps add.
__device__ __forceinline__ void kahan2(float2& s, float2& c, float2 v) {
  float y = v.x - c.x, t = s.x + y;
  c.x = (t - s.x) - y;
  s.x = t;
  y = v.y - c.y;
  t = s.y + y;
  c.y = (t - s.y) - y;
  s.y = t;
}
__device__ __forceinline__ float2 fmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 f2(cd a) { return make_float2(f32_from_f64(a.x), f32_from_f64(a.y)); }

// One source's contribution to the scaled sums of a centre, in the split of
// p2qbxl_pair: sigma^{m+1} A_m and sigma^{m+1} B_m, sigma = 2^s close to k r_c,
// which keeps every term of moderate size. The Hankel recurrence runs in
// float-float on Ht_m = sigma^m H_m,
//   P_m = (2 m sigma / x) Ht_m = sigma^{m+1} K_m,  Z_m = sigma^2 Ht_{m-1},
//   Ht_{m+1} = P_m - Z_m,  sigma^{m+1} E_m = 2 Z_m - P_m,
// everything after it (rounded to FP32) in FP32 with Kahan sums. Real and imaginary
// parts are packed pairs, two operations per issue slot (about 45 slots per order of a
// dipole instead of 72, at two warps per scheduler: 200 ellipses 2.04 -> 1.26 ms, 32
// curves in a batch 5.10 -> 4.22 in all). S: sums, N: their lost parts (the sum is
// S + N). q: sigma times the charge; dn: (d k/2, nu).
template <int PM, bool HS, bool HD>
__device__ __forceinline__ void p2qbxl_pair_mixed(f32p (&S)[2 * PM + 2], f32p (&N)[2 * PM + 2],
                                                  double dx, double dy, float2 q, float4 dn,
                                                  const FfUnits& U, ff c2s, float sg, float sg2,
                                                  int p) {
  FfPolar D;
  if (!D.set(dx, dy, U)) return;
  ffh h0, h1;
  hankel01_ff_any<3>(D.z, h0, h1);
  f32p ph = pk(h0.x.h, h0.y.h), pl = pk(h0.x.l, h0.y.l);  // Ht_{m-1}
  f32p ch = mul2(pk(h1.x.h, h1.y.h), pk(sg, sg));         // Ht_m
  f32p cl = mul2(pk(h1.x.l, h1.y.l), pk(sg, sg));
  const ff c2 = split17(ff_mul_raw(c2s, D.ir));  // 2 sigma / x; m c2.h is exact
  const f32p ah = pk(c2.h, c2.h), al = pk(c2.l, c2.l), nah = pk(-c2.h, -c2.h);
  const f32p z2 = pk(sg2, sg2), nz2 = pk(-sg2, -sg2), nz4 = pk(-2.f * sg2, -2.f * sg2);
  // - D cos psi, D sin psi (psi = th - arg nu)
  f32p dcx = 0, dcy = 0, dsx = 0, dsy = 0, qx = 0, qy = 0;
  auto swap = [](f32p v) {
    const float2 u = unpk(v);
    return pk(u.y, u.x);
  };
  {
    f32p v = N[0];
    if (HS) {
      const f32p h = add2(ph, pl);
      qx = pk(q.x, q.x);
      qy = pk(-q.y, q.y);
      v = fma2(qx, h, fma2(qy, swap(h), v));
    }
    if (HD) {
      const float cpsi = fmaf(D.c, dn.z, D.s * dn.w), spsi = fmaf(D.s, dn.z, -D.c * dn.w);
      const float cx = dn.x * cpsi, cy = dn.y * cpsi, sx = dn.x * spsi, sy = dn.y * spsi;
      dcx = pk(-cx, -cx);
      dcy = pk(cy, -cy);
      dsx = pk(sx, sx);
      dsy = pk(-sy, sy);
      const f32p h = add2(ch, cl), two = pk(2.f, 2.f);
      v = fma2(two, fma2(dcx, h, mul2(dcy, swap(h))), v);  // E_0 = -2 H_1
    }
    kahan_add2(S[0], N[0], v);
  }
  float c = D.c, sn = D.s;  // cos m th, sin m th
  f32p mh = ah, ml = al, nmh = nah;
#pragma unroll
  for (int m = 1; m <= PM; ++m) {
    if (m > p) break;
    if (m > 1) {
      const float t = fmaf(c, D.c, -sn * D.s);
      sn = fmaf(c, D.s, sn * D.c);
      c = t;
      mh = add2(mh, ah);
      nmh = add2(nmh, nah);
      ml = add2(ml, al);
    }
    const f32p cc = pk(c, c), ss = pk(sn, sn);
    // P = (mh + ml) (ch + cl)
    const f32p Ph = mul2(mh, ch);
    const f32p Pl = fma2(ml, ch, fma2(mh, cl, fma2(mh, ch, mul2(nmh, ch))));
    // G = q Ht + D cos psi E, L = D sin psi K: A = G cos + L sin, B = G sin - L cos
    f32p va, vb;
    if (HD) {
      const f32p P = add2(Ph, Pl);
      const f32p E = fma2(add2(ph, pl), nz4, P);  // -E
      f32p G = fma2(dcx, E, mul2(dcy, swap(E)));
      if (HS) {
        const f32p h = add2(ch, cl);
        G = fma2(qx, h, fma2(qy, swap(h), G));
      }
      const f32p L = fma2(dsx, P, mul2(dsy, swap(P)));
      va = fma2(G, cc, fma2(L, ss, N[2 * m]));
      vb = fma2(G, ss, fma2(L, pk(-c, -c), N[2 * m + 1]));
    } else {
      const f32p h = add2(ch, cl);
      const f32p G = fma2(qx, h, mul2(qy, swap(h)));
      va = fma2(G, cc, N[2 * m]);
      vb = fma2(G, ss, N[2 * m + 1]);
    }
    kahan_add2(S[2 * m], N[2 * m], va);
    kahan_add2(S[2 * m + 1], N[2 * m + 1], vb);
    // Ht_{m+1} = P - sigma^2 Ht_{m-1}: the two_sum of the first parts, not renormalised
    const f32p s = fma2(ph, nz2, Ph), t = sub2(s, Ph);
    const f32p e = sub2(sub2(Ph, sub2(s, t)), fma2(ph, z2, t));
    const f32p l = add2(e, fma2(pl, nz2, Pl));
    ph = ch;
    pl = cl;
    ch = s;
    cl = l;
  }
}

// ---------------------------------------------------------------- M2QBXL in mixed precision
// The same translation as m2qbxl_pair_kernel,
//   alpha_l += (-1)^l sum_n mh_n Wh_{n+l} s^{|n| - |n+l|},
// with the Hankel recurrence and the angular factors in FP64 and the Q x P
// products in FP32. The factors span far more than FP32's range (Wh_m grows
// and mh_n falls by many decades with m, n), so each is held in split form,
// FP32 mantissa times 2^e (split_pair): the product of three split factors is
// an FP32 mantissa product and an integer exponent sum, exact apart from the
// FP32 rounding of the mantissas. Every output sums its terms relative to its
// largest one (2^Emax), FP32 with Kahan compensation, and is formed in FP64.
//
// A warp takes PW pairs: lane j runs pair j's recurrence and writes the split
// rows Wp_m = Wh_m e^{i m th}, Wq_m = (-1)^m Wh_m e^{-i m th}, m <= pb + p,
// to shared memory; then the lanes take the warp's (pair, output order)
// items. Inputs: the split multipoles (split_coef_kernel) and the split powers
// s^j, |j| <= p, per level (sf).

// coefficients (multipoles or locals) of every box in split form, same layout
__global__ void split_coef_kernel(const cd* __restrict__ mpole, long long n, float2* __restrict__ mm,
                                int* __restrict__ me) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float2 m;
  int e;
  split_one(mpole[i], m, e);
  mm[i] = m;
  me[i] = e;
}

// s_l^j, j = -p..p, of every level in split form: [n_levels][2p+1]
__global__ void sf_split_kernel(Fmm F, float* __restrict__ sfm, int* __restrict__ sfe) {
  const int l = blockIdx.x, P = 2 * F.p + 1;
  const double* pwl = pw_row(F, l);
  const double* ipl = ipw_row(F, l);
  for (int j = threadIdx.x; j < P; j += blockDim.x) {
    const int jj = j - F.p;
    const double v = jj >= 0 ? pwl[jj] : ipl[-jj];
    float2 m;
    int e;
    split_one(mk(v, 0.0), m, e);
    sfm[(size_t)l * P + j] = m.x;
    sfe[(size_t)l * P + j] = e;
  }
}

__global__ void __launch_bounds__(32) m2qbxl_mixed_kernel(
    Fmm F, const int* __restrict__ pair_ctr, const int* __restrict__ pair_box, int n_pairs,
    int PW, int TW, const float2* __restrict__ mm, const int* __restrict__ me,
    const float* __restrict__ sfm, const int* __restrict__ sfe, cd* __restrict__ partial) {
  extern __shared__ __align__(16) unsigned char m2q_smem[];
  float2* wp = reinterpret_cast<float2*>(m2q_smem);  // [PW][TW]
  float2* wq = wp + (size_t)PW * TW;                 // [PW][TW]
  int* we = reinterpret_cast<int*>(wq + (size_t)PW * TW);  // [PW][TW]
  const int lane = threadIdx.x;
  const int t0 = blockIdx.x * PW;
  const int p = F.p, P = 2 * p + 1;
  const int npw = min(PW, n_pairs - t0);
  if (lane < npw) {
    const int t = t0 + lane;
    const int i = pair_ctr[t], c = pair_box[t];
    const int lc = F.level[c];
    const double s = F.scale[lc];
    const int M = F.lpb[lc] + p;
    const double2 z = F.cxy[i];
    const double2 mc = F.centre[c];
    const double dx = z.x - mc.x, dy = z.y - mc.y;
    const double d2 = dx * dx + dy * dy;
    const double irr = rsqrt(d2), rr = d2 * irr, x = F.k * rr, ix = irr * F.ik;
    const cd e1 = mk(dx * irr, dy * irr);
    cd h0, h1;
    hankel01_wide(x, ix, h0, h1);
    const double c1 = 2.0 * s * ix, s2 = s * s;
    cd hm1 = h0, hm = cscale(h1, s), ee = mk(1.0, 0.0);
    float2* rp = wp + (size_t)lane * TW;
    float2* rq = wq + (size_t)lane * TW;
    int* re = we + (size_t)lane * TW;
    split_pair(h0, h0, rp[0], rq[0], re[0]);
    for (int m = 1; m <= M; ++m) {
      ee = cmul(ee, e1);
      const double ac = hm.x * ee.x, bd = hm.y * ee.y, ad = hm.x * ee.y, bc = hm.y * ee.x;
      const double sm = (m & 1) ? -1.0 : 1.0;
      split_pair(mk(ac - bd, ad + bc), mk(sm * (ac + bd), sm * (bc - ad)), rp[m], rq[m], re[m]);
      const cd hn = mk(fma((double)m * c1, hm.x, -s2 * hm1.x), fma((double)m * c1, hm.y, -s2 * hm1.y));
      hm1 = hm;
      hm = hn;
    }
  }
  __syncwarp();
  for (int o = lane; o < npw * P; o += 32) {
    const int u = o / P, lo = o % P - p;
    const int t = t0 + u;
    const int c = pair_box[t];
    const int lc = F.level[c];
    const int pb = F.lpb[lc];
    const long long off = F.eoff[c] + pb;
    const float2* rp = wp + (size_t)u * TW;
    const float2* rq = wq + (size_t)u * TW;
    const int* re = we + (size_t)u * TW;
    const float* fm = sfm + (size_t)lc * P + p;
    const int* fe = sfe + (size_t)lc * P + p;
    // one pass: the sums are kept relative to the largest exponent seen so
    // far and rescaled (by a power of two) when a larger one appears
    int emax = 2 * kZeroExp;
    float2 S = make_float2(0.f, 0.f), C = make_float2(0.f, 0.f);
    for (int n = -pb; n <= pb; ++n) {
      const int m = n + lo, am = abs(m);
      const int j = abs(n) - am;
      const int e = me[off + n] + re[am] + fe[j];
      if (e > emax) {
        const float r = pow2f(emax - e);
        S = make_float2(S.x * r, S.y * r);
        C = make_float2(C.x * r, C.y * r);
        emax = e;
      }
      const int d = e - emax;
      if (d < -126) continue;
      const float f = fm[j] * pow2f(d);
      const float2 w = m >= 0 ? rp[am] : rq[am];
      const float2 v = fmul(mm[off + n], w);
      kahan2(S, C, make_float2(v.x * f, v.y * f));
    }
    const double sc = (lo & 1) ? -pow2d(emax) : pow2d(emax);
    partial[(size_t)t * P + lo + p] =
        mk(((double)S.x - (double)C.x) * sc, ((double)S.y - (double)C.y) * sc);
  }
}

// ---------------------------------------------------------------- L2QBXL in mixed precision
// The translation of l2qbxl_kernel, alpha_s += sum_n gamma_n t_{s-n}, with the
// Miller recurrence (J_m) and the angular factors in FP64 and the products in
// FP32 on split factors (as in m2qbxl_mixed_kernel): the leaf's local
// coefficients gamma_n (large for large |n|) and the row V_m = J_m e^{i m th}
// (small for large m) as FP32 mantissas with integer exponents; each output
// sums relative to its largest term with Kahan compensation. A warp takes G
// centres; lane j fills centre j's row in FP64 and converts it in place to
// split form (FP32 mantissa pair and exponent in the 16 bytes of each entry).
__global__ void __launch_bounds__(32) l2qbxl_mixed_kernel(Fmm F, const int* __restrict__ cleaf,
                                                          const int* __restrict__ clist, int n_ctr,
                                                          int G, int TW,
                                                          const float2* __restrict__ gm,
                                                          const int* __restrict__ ge,
                                                          cd* __restrict__ alpha) {
  extern __shared__ cd trow[];  // [G][TW]
  const int lane = threadIdx.x;
  const int c0 = blockIdx.x * G;
  const int p = F.p, P = 2 * p + 1;
  if (lane < G && c0 + lane < n_ctr) {
    const int i = clist[c0 + lane];
    const int b = cleaf[i];
    const int M = F.lpb[F.level[b]] + p;
    const double2 mb = F.centre[b];
    const double dx = F.cxy[i].x - mb.x, dy = F.cxy[i].y - mb.y;
    const double rr = sqrt(dx * dx + dy * dy);
    cd* row = trow + (size_t)lane * TW;
    const double in = 1.0 / miller_row(F.k * rr, M, (double*)row, 2);
    const cd e1 = rr > 0.0 ? mk(dx / rr, dy / rr) : mk(1.0, 0.0);
    cd e = mk(1.0, 0.0);
    for (int m = 0; m <= M; ++m) {
      float2 mv;
      int ev;
      split_one(cscale(e, row[m].x * in), mv, ev);
      float4* slot = reinterpret_cast<float4*>(row + m);
      *slot = make_float4(mv.x, mv.y, __int_as_float(ev), 0.f);
      e = cmul(e, e1);
    }
  }
  __syncwarp();
  const int nG = min(G, n_ctr - c0);
  for (int o = lane; o < nG * P; o += 32) {
    const int u = o / P, so = o % P - p;
    const int i = clist[c0 + u];
    const int b = cleaf[i];
    const int pb = F.lpb[F.level[b]];
    const float4* row = reinterpret_cast<const float4*>(trow + (size_t)u * TW);
    const long long off = F.eoff[b] + pb;
    // one pass: the sums are kept relative to the largest exponent seen so
    // far and rescaled (by a power of two) when a larger one appears
    int emax = 2 * kZeroExp;
    float2 S = make_float2(0.f, 0.f), C = make_float2(0.f, 0.f);
    for (int n = -pb; n <= pb; ++n) {
      const int m = so - n;
      const float4 v = row[abs(m)];
      const int e = ge[off + n] + __float_as_int(v.z);
      if (e > emax) {
        const float r = pow2f(emax - e);
        S = make_float2(S.x * r, S.y * r);
        C = make_float2(C.x * r, C.y * r);
        emax = e;
      }
      const int d = e - emax;
      if (d < -126) continue;
      // t_m = (-1)^m V_m (m >= 0), conj(V_-m) (m < 0): signs on the bits
      const unsigned fx = (m >= 0 && (m & 1)) ? 0x80000000u : 0u;
      const unsigned fy = m < 0 ? 0x80000000u : fx;
      const float2 t = make_float2(__uint_as_float(__float_as_uint(v.x) ^ fx),
                                   __uint_as_float(__float_as_uint(v.y) ^ fy));
      const float f = pow2f(d);
      const float2 w = fmul(gm[off + n], t);
      kahan2(S, C, make_float2(w.x * f, w.y * f));
    }
    const double sc = pow2d(emax);
    cd* dst = alpha + (size_t)F.cid[i] * P + p + so;
    *dst = cadd(*dst, cscale2(mk(((double)S.x - (double)C.x) * sc, ((double)S.y - (double)C.y) * sc),
                              out_exp(F)));
  }
}

// ---------------------------------------------------------------- L2QBXL, M2QBXL on float-float levels
// The two translations above when every leaf (W-list box) of the launch is on a
// level with a power-of-two scaling s = ffs (almost always): the scaled
// coefficients and rows fit FP32, so a term is a plain FP32 product and no
// exponents are carried. With g_n = 2^{s|n|} gamma_n and v_m = 2^{-s|m|} V_m,
//   alpha_l = 2^{-s|l|} sum_n g_n t_{l-n} 2^{s(|l-n| - |n| + |l|)},
// and for n' = n sgn(l) the exponent is 2 s |l| for n' <= 0 and 2 s max(|l| - n', 0)
// for n' > 0: two Kahan sums, joined in FP64. M2QBXL has the same form with the
// roles of the sides exchanged. Rows by the float-float recurrences; angular
// factors FP32 between float-float anchors every eighth order. (200 ellipses: L2QBXL
// 1.02 -> 0.47 ms, M2QBXL 0.67 -> 0.24, against the FP64 rows and split exponents.)
__global__ void __launch_bounds__(32) l2qbxl_ff_kernel(Fmm F, const int* __restrict__ cleaf,
                                                       const int* __restrict__ clist, int n_ctr,
                                                       int G, int TW, cd* __restrict__ alpha) {
  extern __shared__ __align__(16) float2 frow[];  // [G][TW], TW = max M + 1
  const int lane = threadIdx.x;
  const int c0 = blockIdx.x * G;
  const int p = F.p, P = 2 * p + 1;
  if (lane < G && c0 + lane < n_ctr) {
    const int i = clist[c0 + lane];
    const int b = cleaf[i];
    const int l = F.level[b], M = F.lpb[l] + p, s = F.ffs[l];
    const double2 mb = F.centre[b], z = F.cxy[i];
    const FfUnits& U = F.U;
    FfPolar D;
    const bool off = D.set(z.x - mb.x, z.y - mb.y, U);
    float2* row = frow + (size_t)lane * TW;
    if (!off || D.z.h < 1e-8f) {  // J_m(x) = (x/2)^m / m!
      float t = 1.f;
      const float hx = off ? 0.5f * D.z.h * pow2f(-s) : 0.f;
      float2 e = make_float2(1.f, 0.f);
      for (int m = 0; m <= M; ++m) {
        row[m] = make_float2(e.x * t, e.y * t);
        t *= hx / (float)(m + 1);
        if (off) e = fmul(e, make_float2(D.c, D.s));
      }
    } else {
      const ff inv = ff_miller_row(row, M, s, D, U);
      const ff c1 = ff_mul(D.x, D.ir), s1 = ff_mul(D.y, D.ir);
      ff c8 = c1, s8 = s1;
#pragma unroll
      for (int u = 0; u < 3; ++u) ff_turn(c8, s8, c8, s8);
      const float2 e1 = make_float2(ff_f32(c1), ff_f32(s1));
      ff ex = mkff(1.f, 0.f), ey = mkff(0.f, 0.f);
      float2 e = make_float2(1.f, 0.f);
      float sc = 1.f;
      for (int m = 0; m <= M; ++m) {
        if ((m & 7) == 0) {
          e = make_float2(ff_f32(ex), ff_f32(ey));
          ff_turn(ex, ey, c8, s8);
        } else {
          e = fmul(e, e1);
        }
        const float v = ff_f32(ff_mul_raw(ff_miller_value(row[m], sc), inv));
        row[m] = make_float2(e.x * v, e.y * v);
      }
    }
  }
  __syncwarp();
  const int nG = min(G, n_ctr - c0);
  for (int o = lane; o < nG * P; o += 32) {
    const int u = o / P, so = o % P - p;
    const int i = clist[c0 + u];
    const int b = cleaf[i];
    const int l = F.level[b], pb = F.lpb[l], s = F.ffs[l];
    const float2* row = frow + (size_t)u * TW;
    const float2* g = F.loc32 + F.eoff[b] + pb;
    const int a = abs(so), dir = so < 0 ? -1 : 1;
    // t_m = (-1)^m V_m for m >= 0, conj(V_{-m}) for m < 0 (signs on the bits)
    auto term = [](float2 gn, float2 v, bool neg, int m) {
      const unsigned fx = !neg && (m & 1) ? 0x80000000u : 0u;
      const unsigned fy = neg ? 0x80000000u : fx;
      return fmul(gn, make_float2(__uint_as_float(__float_as_uint(v.x) ^ fx),
                                  __uint_as_float(__float_as_uint(v.y) ^ fy)));
    };
    float2 S1 = make_float2(0.f, 0.f), C1 = S1, S2 = S1, C2 = S1;
    for (int j = 0; j <= pb; ++j)  // n' = -j: m = dir (a + j)
      kahan2(S1, C1, term(g[-dir * j], row[a + j], so < 0, a + j));
    for (int j = 1; j <= pb; ++j) {  // n' = j: m = dir (a - j)
      const int m = abs(a - j);
      const bool neg = (a > j) ? so < 0 : (a < j) ? so >= 0 : false;
      float2 v = term(g[dir * j], row[m], neg, m);
      if (j < a) {
        const float f = pow2f(2 * s * (a - j));
        v = make_float2(v.x * f, v.y * f);
      }
      kahan2(S2, C2, v);
    }
    const double f1 = pow2d(s * a), f2 = pow2d(-s * a);
    cd* dst = alpha + (size_t)F.cid[i] * P + p + so;
    const cd v = mk(((double)S1.x - (double)C1.x) * f1 + ((double)S2.x - (double)C2.x) * f2,
                    ((double)S1.y - (double)C1.y) * f1 + ((double)S2.y - (double)C2.y) * f2);
    *dst = cadd(*dst, cscale2(v, out_exp(F)));
  }
}

// a_n 2^{-s|n|} in FP32 of the boxes listed (a_n = mh_n s_l^|n|), for M2QBXL
__global__ void __launch_bounds__(kThreads) mpole_scaled_kernel(Fmm F, const int* __restrict__ boxes,
                                                                float2* __restrict__ out) {
  const int b = boxes[blockIdx.x];
  const int l = F.level[b], pb = F.lpb[l], s = F.ffs[l];
  const double* pwl = pw_row(F, l);
  const cd* a = F.mpole + F.eoff[b] + pb;
  float2* dst = out + F.eoff[b] + pb;
  for (int n = (int)threadIdx.x - pb; n <= pb; n += kThreads) {
    const double f = pwl[abs(n)];
    dst[n] = make_float2(f32_from_f64_sh(a[n].x * f, -s * abs(n)),
                         f32_from_f64_sh(a[n].y * f, -s * abs(n)));
  }
}

// M2QBXL: alpha_l += (-1)^l sum_n a_n W_{n+l} over (centre, W box) pairs, PW per
// warp. With A_n = 2^{-s|n|} a_n, w_m = 2^{s|m|} W_m and n' = n sgn(l) the exponent
// of a term is -s|l| plus 0 for n' >= 0 and 2 s min(-n', |l|) for n' < 0.
__global__ void __launch_bounds__(32) m2qbxl_ff_kernel(
    Fmm F, const int* __restrict__ pair_ctr, const int* __restrict__ pair_box, int n_pairs, int PW,
    int TW, const float2* __restrict__ A, cd* __restrict__ partial) {
  extern __shared__ __align__(16) float4 qrow[];  // [PW][TW]: w_m, w_{-m}
  const int lane = threadIdx.x;
  const int t0 = blockIdx.x * PW;
  const int p = F.p, P = 2 * p + 1;
  const int npw = min(PW, n_pairs - t0);
  if (lane < npw) {
    const int i = pair_ctr[t0 + lane], c = pair_box[t0 + lane];
    const int l = F.level[c], M = F.lpb[l] + p, s = F.ffs[l];
    const double2 z = F.cxy[i], mc = F.centre[c];
    const FfUnits& U = F.U;
    FfPolar D;
    D.set(z.x - mc.x, z.y - mc.y, U);
    ffh hp, hc;
    hankel01_ff_any<3>(D.z, hp, hc);
    const float sg = pow2f(s), sg2 = pow2f(2 * s);
    hc.x = ff_scale(hc.x, sg);
    hc.y = ff_scale(hc.y, sg);
    const ff c2 = split17(ff_mul_raw(ff_scale(U.ik2, sg), D.ir));  // 2 2^s / x
    const ff c1 = ff_mul(D.x, D.ir), s1 = ff_mul(D.y, D.ir);
    ff c8 = c1, s8 = s1;
#pragma unroll
    for (int u = 0; u < 3; ++u) ff_turn(c8, s8, c8, s8);
    const float2 e1 = make_float2(ff_f32(c1), ff_f32(s1));
    ff ex = c8, ey = s8;
    float2 e = e1;
    float4* row = qrow + (size_t)lane * TW;
    const float2 h0 = make_float2(ff_f32(hp.x), ff_f32(hp.y));
    row[0] = make_float4(h0.x, h0.y, h0.x, h0.y);
    for (int m = 1; m <= M; ++m) {
      if ((m & 7) == 0) {
        e = make_float2(ff_f32(ex), ff_f32(ey));
        ff_turn(ex, ey, c8, s8);
      } else if (m > 1) {
        e = fmul(e, e1);
      }
      const float2 hm = make_float2(ff_f32(hc.x), ff_f32(hc.y));
      const float2 wp = fmul(hm, e), wq = fmul(hm, make_float2(e.x, -e.y));
      row[m] = (m & 1) ? make_float4(wp.x, wp.y, -wq.x, -wq.y) : make_float4(wp.x, wp.y, wq.x, wq.y);
      const ff cm = mkff((float)m * c2.h, (float)m * c2.l);
      const ff nx = ff_sub_raw(ff_mul_raw(cm, hc.x), ff_scale(hp.x, sg2));
      const ff ny = ff_sub_raw(ff_mul_raw(cm, hc.y), ff_scale(hp.y, sg2));
      hp = hc;
      hc.x = nx;
      hc.y = ny;
    }
  }
  __syncwarp();
  for (int o = lane; o < npw * P; o += 32) {
    const int u = o / P, lo = o % P - p;
    const int c = pair_box[t0 + u];
    const int l = F.level[c], pb = F.lpb[l], s = F.ffs[l];
    const float4* row = qrow + (size_t)u * TW;
    const float2* an = A + F.eoff[c] + pb;
    const int a = abs(lo), dir = lo < 0 ? -1 : 1;
    auto w = [&](int m, bool neg) {
      const float4 v = row[m];
      return neg ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
    };
    float2 S1 = make_float2(0.f, 0.f), C1 = S1, S2 = S1, C2 = S1;
    for (int j = 0; j <= pb; ++j)  // n' = j: m = dir (a + j)
      kahan2(S1, C1, fmul(an[dir * j], w(a + j, lo < 0)));
    for (int j = 1; j <= pb; ++j) {  // n' = -j: m = dir (a - j)
      const bool neg = (a > j) ? lo < 0 : lo >= 0;
      const float2 v = fmul(an[-dir * j], w(abs(a - j), neg));
      if (j < a) {  // the exponent grows from n' = 0's by 2 s j (s < 0)
        const float f = pow2f(2 * s * j);
        kahan2(S1, C1, make_float2(v.x * f, v.y * f));
      } else {
        kahan2(S2, C2, v);
      }
    }
    // exponents -s a for n' > -a (after the factors), s a for n' <= -a
    double f1 = pow2d(-s * a), f2 = pow2d(s * a);
    if (lo & 1) f1 = -f1, f2 = -f2;
    partial[(size_t)(t0 + u) * P + lo + p] =
        mk(((double)S1.x - (double)C1.x) * f1 + ((double)S2.x - (double)C2.x) * f2,
           ((double)S1.y - (double)C1.y) * f1 + ((double)S2.y - (double)C2.y) * f2);
  }
}

// ---------------------------------------------------------------- P2P in mixed precision
// p2p_warp_kernel with everything but the two coordinate differences in
// float-float (strengths, normals, tables to degree-6 second parts, the lanes'
// sums; the warp's sum is FP64): about 300 FP32 instructions per source and
// layer in place of 45 on the FP64 pipe, which bound it (82 % of its rate): 11 M
// pairs of 200 ellipses 1.22 -> 0.26 ms, the starfish grid 0.19 -> 0.05 ms.
struct FfSum {
  ff x, y;
  __device__ __forceinline__ FfSum() : x(mkff(0.f, 0.f)), y(mkff(0.f, 0.f)) {}
  // += a b, complex a given as (re h, re l, im h, im l)
  __device__ __forceinline__ void fma(float4 a, ff bx, ff by) {
    const ff ax = mkff(a.x, a.y), ay = mkff(a.z, a.w);
    x = ff_add(x, ff_sub_raw(ff_mul_raw(ax, bx), ff_mul_raw(ay, by)));
    y = ff_add(y, ff_sub_raw(ff_mul_raw(ax, by), ff_mul_raw(mkff(-ay.h, -ay.l), bx)));
  }
};

template <bool HS, bool HD>
__global__ void __launch_bounds__(kThreads) p2p_warp_mixed_kernel(Fmm F, const int* __restrict__ utgt,
                                                                  const int* __restrict__ tleaf,
                                                                  int n, cd* __restrict__ out) {
  const int t = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (t >= n) return;
  const int i = utgt[t];
  const int b = tleaf[i];
  const double2 tp = F.txy[i];
  const FfUnits& U = F.U;
  FfSum acc;
  const SourceCursor sc{F.uidx, F.rsrc, F.uoff[b], F.uoff[b + 1] - F.uoff[b], 0, 0, nullptr};
  deal_sources(sc, lane, [&](int j) {
    const double2 y = F.sxy[j];
    FfPolar D;
    if (!D.set(tp.x - y.x, tp.y - y.y, U)) return;
    ffh h0, h1;
    hankel01_ff_any<kHankLoFf, HS, HD>(D.z, h0, h1);
    if (HS) acc.fma(F.qf[j], h0.x, h0.y);
    if (HD) {
      const float4 nv = F.nf[j];  // n . (t - y) / r
      const ff f = ff_mul(ff_add(ff_mul_raw(mkff(nv.x, nv.y), D.x),
                                 ff_mul_raw(mkff(nv.z, nv.w), D.y)), D.ir);
      acc.fma(F.df[j], ff_mul_raw(h1.x, f), ff_mul_raw(h1.y, f));
    }
  });
  cd sum = mk(ff_f64(acc.x), ff_f64(acc.y));
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    sum.x += __shfl_xor_sync(0xffffffffu, sum.x, off);
    sum.y += __shfl_xor_sync(0xffffffffu, sum.y, off);
  }
  if (lane == 0) {
    cd* dst = out + F.tid[i];
    *dst = cadd(*dst, cscale2(sum, out_exp(F)));
  }
}

// ---------------------------------------------------------------- L2P in mixed precision
// l2p_kernel's Miller and Clenshaw recurrences in float-float, on 2^{-s m} J_m
// and the coefficients scaled by 2^{s m} (s = ffs of the level):
//   f_{n-1} = (2 n 2^s / x) f_n - 4^s f_{n+1},  norm = f_0 + 2 4^s (f_2 + 4^s (f_4 + ...)),
// everything kept rescaled by 2^-60 when |f| passes 2^20: the coefficients are sums of
// strengths below 2 times Hankel values below 2^60 (float_float_scale), which leaves
// 2^47 for the number of sources. About 110 FP32 instructions per
// order instead of 11 on the FP64 pipe, which bound it (86 % of its rate): 0.9 M
// targets of 200 ellipses 1.75 -> 0.32 ms.
// Levels without a scale and targets within x = 1e-8 of the centre take the
// FP64 form, out of line.
static __device__ __noinline__ void l2p_value_outside(const Fmm& F, int i, int b, cd* v) {
  *v = l2p_value(F, i, b);
}

__global__ void __launch_bounds__(kThreads) l2p_mixed_kernel(Fmm F, const int* __restrict__ dtgt,
                                                             const int* __restrict__ tleaf, int n,
                                                             cd* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int i = dtgt[t];
  const int b = tleaf[i];
  const int l = F.level[b];
  const int pb = F.lpb[l], s = F.ffs[l];
  cd* dst = out + F.tid[i];
  const double2 mc = F.centre[b], tp = F.txy[i];
  const FfUnits& U = F.U;
  FfPolar D;
  const bool in = s != kNoFf && D.set(tp.x - mc.x, tp.y - mc.y, U) && D.z.h >= 1e-8f;
  if (!in) {
    cd v;
    l2p_value_outside(F, i, b, &v);
    *dst = cadd(*dst, cscale2(v, out_exp(F)));
    return;
  }
  const float4* pq = reinterpret_cast<const float4*>(F.lpq + F.eoff[b]);
  const float sg2 = pow2f(2 * s);
  ff c2 = ff_mul_raw(ff_scale(U.ik2, pow2f(s)), D.ir);  // 2 2^s / x
  c2 = fast_two_sum(c2.h, c2.l);
  const ff co = ff_mul(D.x, D.ir), si = ff_mul(D.y, D.ir);
  const ff co2 = ff_scale(co, 2.f);
  const int N = miller_start_f32(pb, D.z.h);
  ff f1 = mkff(0.f, 0.f), f0 = mkff(0x1p-40f, 0.f), sum = f1;
  float fn = (float)N;
  auto step = [&]() {
    const float ch = __fmul_rn(fn, c2.h);
    const ff cn = mkff(ch, __fmaf_rn(fn, c2.l, __fmaf_rn(fn, c2.h, -ch)));
    const ff f = ff_sub_raw(ff_mul_raw(cn, f0), ff_scale(f1, sg2));
    f1 = f0;
    f0 = fast_two_sum(f.h, f.l);
    fn -= 1.f;
  };
  auto even = [&]() { sum = ff_add(f0, ff_scale(sum, sg2)); };
  constexpr float kBig = 0x1p20f, kDown = 0x1p-60f;
  int nn = N;
  for (; nn >= pb + 2; --nn) {  // orders above pb: the recurrence alone
    if ((nn & 1) == 0) even();
    step();
    if (fabsf(f0.h) >= kBig) {
      f0 = ff_scale(f0, kDown);
      f1 = ff_scale(f1, kDown);
      sum = ff_scale(sum, kDown);
    }
  }
  // one Clenshaw step of a real component: f c + 2 cos(th) b1 - b2
  auto clenshaw = [&](ff c, ff& b1, ff& b2) {
    const ff p = ff_mul_raw(f0, c), q = ff_mul_raw(co2, b1);
    const ff u = two_sum(q.h, -b2.h), v = two_sum(u.h, p.h);
    const float lo = __fadd_rn(__fadd_rn(u.l, v.l), __fadd_rn(p.l, __fsub_rn(q.l, b2.l)));
    b2 = b1;
    b1 = fast_two_sum(v.h, lo);
  };
  const ff z = mkff(0.f, 0.f);
  ff ux1 = z, ux2 = z, uy1 = z, uy2 = z, vx1 = z, vx2 = z, vy1 = z, vy2 = z;
  for (; nn >= 1; --nn) {
    if ((nn & 1) == 0) even();
    step();
    const int mm = nn - 1;  // f0 = f_mm
    const float4 P = pq[mm];
    clenshaw(mkff(P.x, P.y), ux1, ux2);
    clenshaw(mkff(P.z, P.w), uy1, uy2);
    if (mm >= 1) {
      const float4 Q = pq[pb + mm];
      clenshaw(mkff(Q.x, Q.y), vx1, vx2);
      clenshaw(mkff(Q.z, Q.w), vy1, vy2);
    }
    if (fabsf(f0.h) >= kBig) {
      ff* const kept[] = {&f0, &f1, &sum, &ux1, &ux2, &uy1, &uy2, &vx1, &vx2, &vy1, &vy2};
#pragma unroll
      for (ff* v : kept) *v = ff_scale(*v, kDown);
    }
  }
  const ff norm = ff_add(f0, ff_scale(sum, 2.f * sg2));
  // u_0 - cos(th) u_1 + sin(th) v_1, over norm
  auto finish = [&](ff u1, ff u2, ff v1) {
    return ff_add(ff_add(u1, ff_mul(mkff(-co.h, -co.l), u2)), ff_mul(si, v1));
  };
  const double in64 = scale2(1.0 / ff_f64(norm), out_exp(F));
  const ff ax = finish(ux1, ux2, vx1), ay = finish(uy1, uy2, vy1);
  *dst = cadd(*dst, mk(ff_f64(ax) * in64, ff_f64(ay) * in64));
}

// ---------------------------------------------------------------- M2P in mixed precision
// The FP32 multipoles that M2P reads, at entry eoff[b] + b of a float2 array
// (2 pb + 2 entries per box). On float-float levels (ffs[l] = s)
// box b holds float4 (P_m, Q_m), m = 0..pb, of the term of order m
//   a_m H_m e^{i m th} + a_{-m} H_{-m} e^{-i m th} = H_m (P_m cos m th + Q_m sin m th),
//   P_m = a_m + (-1)^m a_{-m},  Q_m = i (a_m - (-1)^m a_{-m}),  P_0 = a_0,
// times 2^{-s m} (a_n = mh_n s_l^|n| the true coefficient); on the other levels
// the sigma-normalised mu_n = mh_n conv_|n| (conv = s^j / sig_j), n = -pb..pb.
__global__ void __launch_bounds__(kThreads) mpole_f32_list_kernel(
    Fmm F, const int* __restrict__ boxes, const double* __restrict__ conv,
    float2* __restrict__ mu) {
  const int b = boxes[blockIdx.x];
  const int l = F.level[b];
  const int pb = F.lpb[l];
  const int s = F.ffs[l];
  const cd* a = F.mpole + F.eoff[b] + pb;
  float2* dst = mu + F.eoff[b] + b;
  if (s == kNoFf) {
    const double* cv = conv + (size_t)l * (F.pbmax + 1);
    for (int n = (int)threadIdx.x - pb; n <= pb; n += kThreads) {
      const double f = cv[abs(n)];
      dst[n + pb] = make_float2((float)(a[n].x * f), (float)(a[n].y * f));
    }
    return;
  }
  const double* pwl = pw_row(F, l);
  for (int m = threadIdx.x; m <= pb; m += kThreads) {
    // the power of two, up to 2^1500, as an exponent offset
    const int sh = -s * m;
    const double f = pwl[m];
    cd g = m > 0 ? a[-m] : mk(0.0, 0.0);
    if (m & 1) g = mk(-g.x, -g.y);
    const cd P = cscale(cadd(a[m], g), f), d = cscale(csub(a[m], g), f);
    reinterpret_cast<float4*>(dst)[m] =
        make_float4(f32_from_f64_sh(P.x, sh), f32_from_f64_sh(P.y, sh),
                    m ? f32_from_f64_sh(-d.y, sh) : 0.f, m ? f32_from_f64_sh(d.x, sh) : 0.f);
  }
}

// M2P: a thread per (direct target, W-list box) pair, pairs ordered by (leaf,
// box, target) so that the lanes of a warp read the same box's coefficients;
// slot[t] is the pair's place in target order, where m2p_sum_mixed_kernel adds.
//  * float-float levels: Ht_m = 2^{s m} H_m(k r) by the float-float recurrence
//      Ht_{m+1} = (2 m 2^s / x) Ht_m - 4^s Ht_{m-1};
//  * levels whose orders do not fit FP32's range that way (hundreds of orders
//    over boxes of many wavelengths): G_m = sig_m H_m in FP64 by
//      G_{m+1} = (2m/x)(sig_{m+1}/sig_m) G_m - (sig_{m+1}/sig_{m-1}) G_{m-1}
//    (rec[l][m] = (2m sig_{m+1}/sig_m, sig_{m+1}/sig_{m-1}), rec[l][0].x =
//    sig_1) against mu_m = a_m / sig_m.
// Angular factors, products and the compensated (Kahan) sum are FP32. With the
// recurrence in FP64 on every level the kernel ran at 87 % of the FP64 pipe (4.8 M
// pairs of 200 ellipses: 2.11 -> 0.76 ms; with packed pairs and the pairs' sums joined
// in float-float 0.62; with the multipoles rounded by integer instructions 0.57).
__global__ void __launch_bounds__(kThreads) m2p_pair_mixed_kernel(
    Fmm F, const int* __restrict__ pt, const int* __restrict__ pbx, const int* __restrict__ slot,
    int n, const float2* __restrict__ mu, const double2* __restrict__ rec,
    float4* __restrict__ partial) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int i = pt[t], c = pbx[t];
  const int lc = F.level[c];
  const int pb = F.lpb[lc];
  const int s = F.ffs[lc];
  const double2 mc = F.centre[c];
  const double dx = F.txy[i].x - mc.x, dy = F.txy[i].y - mc.y;
  float2 S, C = make_float2(0.f, 0.f);  // the sum is S - C
  if (s != kNoFf) {  // packed (re, im) pairs, as in p2qbxl_pair_mixed
    const ulonglong2* a = reinterpret_cast<const ulonglong2*>(mu + F.eoff[c] + c);  // (P_m, Q_m)
    const FfUnits& U = F.U;
    FfPolar D;
    D.set(dx, dy, U);
    ffh h0, h1;
    hankel01_ff_any<3>(D.z, h0, h1);
    const float sg = pow2f(s), sg2 = pow2f(2 * s);
    const ff c2 = split17(ff_mul_raw(ff_scale(U.ik2, sg), D.ir));  // 2 2^s / x
    f32p ph = pk(h0.x.h, h0.y.h), pl = pk(h0.x.l, h0.y.l);
    f32p ch = mul2(pk(h1.x.h, h1.y.h), pk(sg, sg)), cl = mul2(pk(h1.x.l, h1.y.l), pk(sg, sg));
    const f32p ah = pk(c2.h, c2.h), al = pk(c2.l, c2.l), nah = pk(-c2.h, -c2.h);
    const f32p z2 = pk(sg2, sg2), nz2 = pk(-sg2, -sg2);
    const float2 p0 = unpk(a[0].x), w0 = unpk(add2(ph, pl));
    const float2 v0 = fmul(p0, w0);
    f32p sum = pk(v0.x, v0.y), lost = 0ull;
    float co = D.c, si = D.s;
    f32p mh = ah, ml = al, nmh = nah;
    for (int m = 1; m <= pb; ++m) {
      const ulonglong2 pq = a[m];
      const float2 v = unpk(fma2(pq.x, pk(co, co), mul2(pq.y, pk(si, si))));
      const f32p h = add2(ch, cl);
      const float2 u = unpk(h);
      kahan_add2(sum, lost, fma2(pk(v.x, v.x), h, fma2(pk(-v.y, v.y), pk(u.y, u.x), lost)));
      const f32p Ph = mul2(mh, ch);
      const f32p Pl = fma2(ml, ch, fma2(mh, cl, fma2(mh, ch, mul2(nmh, ch))));
      const f32p t1 = fma2(ph, nz2, Ph), t2 = sub2(t1, Ph);
      const f32p e = sub2(sub2(Ph, sub2(t1, t2)), fma2(ph, z2, t2));
      const f32p l = add2(e, fma2(pl, nz2, Pl));
      ph = ch;
      pl = cl;
      ch = t1;
      cl = l;
      mh = add2(mh, ah);
      nmh = add2(nmh, nah);
      ml = add2(ml, al);
      const float t = fmaf(co, D.c, -si * D.s);
      si = fmaf(co, D.s, si * D.c);
      co = t;
    }
    S = unpk(sum);
    C = unpk(lost);
    C = make_float2(-C.x, -C.y);
  } else {
    const float2* a = mu + F.eoff[c] + c + pb;  // a[m], |m| <= pb
    const double d2 = dx * dx + dy * dy;
    const double irr = rsqrt(d2), rr = d2 * irr, x = F.k * rr, ix = irr * F.ik;
    cd h0, h1;
    hankel01_wide(x, ix, h0, h1);
    const float irf = f32_from_f64(irr);
    const float2 e1 = make_float2(f32_from_f64(dx) * irf, f32_from_f64(dy) * irf);
    float2 ee = e1;
    S = fmul(a[0], f2(h0));
    const double2* R = rec + (size_t)lc * (F.pbmax + 2);
    cd gprev = h0, gcur = cscale(h1, R[0].x);
    for (int m = 1; m <= pb; ++m) {
      const float2 g = f2(gcur);
      const float2 wp = fmul(g, ee);                                // G_m e^{im th}
      float2 wn = fmul(g, make_float2(ee.x, -ee.y));                // G_m e^{-im th}
      if (m & 1) wn = make_float2(-wn.x, -wn.y);                    // (-1)^m
      const float2 vp = fmul(a[m], wp), vn = fmul(a[-m], wn);
      kahan2(S, C, make_float2(vp.x + vn.x, vp.y + vn.y));
      if (m < pb) {
        const double c1 = R[m].x * ix, c2 = R[m].y;
        const cd gn = mk(fma(c1, gcur.x, -c2 * gprev.x), fma(c1, gcur.y, -c2 * gprev.y));
        gprev = gcur;
        gcur = gn;
        ee = fmul(ee, e1);
      }
    }
  }
  partial[slot[t]] = make_float4(S.x, -C.x, S.y, -C.y);
}

// out[target] += sum of its pairs' float-float terms, in pair order.
__global__ void m2p_sum_mixed_kernel(int n, const int* __restrict__ wtgt, const int* __restrict__ off,
                                     const float4* __restrict__ partial, const int* __restrict__ tid,
                                     const int* __restrict__ sexp, cd* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  ff x = mkff(0.f, 0.f), y = x;
  for (int e = off[t]; e < off[t + 1]; ++e) {
    const float4 v = partial[e];
    x = ff_add(x, mkff(v.x, v.y));
    y = ff_add(y, mkff(v.z, v.w));
  }
  cd* dst = out + tid[wtgt[t]];
  *dst = cadd(*dst, cscale2(mk(ff_f64(x), ff_f64(y)), *sexp));
}

// ---------------------------------------------------------------- P2M in mixed precision
// The item structure of p2m_item_kernel with rows and sums in FP32:
// R_t = conj(V_t) / sig_|t| and, over the item's sources with Kahan compensation,
//   mu_n = sum_j [q_j R_n + A_j R_{n-1} sig_|n-1| / sig_|n| - B_j R_{n+1} sig_|n+1| / sig_|n|],
// A = d (k/2) conj(nu), B = d (k/2) nu; mu_n = a_n / sig_|n|, of order one.
// p2m_sum_mixed_kernel adds a leaf's segments in FP64 and forms mh_n = mu_n /
// conv_|n| (conv = s^j / sig_j).
// Row of source i for a box of level l with centre m: row[t] = R_t, 0 <= t <= pb + 1
// (R_{-t} = (-1)^t conj(R_t)). On float-float levels the Miller recurrence of
// l2p_mixed_kernel on 2^{-s j} J_j (its values kept in the row while it runs),
// normalised and brought to J_j / sig_j by isf[j] = 2^{s j} / sig_j; elsewhere in
// FP64, one product per order, the normalisation as an exponent offset and an
// FP32 factor. The angular factors e^{-i j th} are FP32 products between
// float-float anchors every eighth order. (One warp fills an item's rows while the
// others wait, so the FP64 recurrence's rate set the kernel's: 2^20 sources in 200
// ellipses 1.25 -> 0.84 ms.)
__device__ __forceinline__ void p2m_fill_row_mixed(const Fmm& F, const FfUnits& U, int i, double2 m,
                                                   int l, int pb, float2* row) {
  const double2 y = F.sxy[i];
  FfPolar D;
  const bool off = D.set(y.x - m.x, y.y - m.y, U);
  const int s = F.ffs[l];
  const bool in = s != kNoFf && off && D.z.h >= 1e-8f;
  ff inv = mkff(0.f, 0.f);
  int en = 0;
  float imn = 0.f;
  if (in) {
    inv = ff_miller_row(row, pb + 1, s, D, U);
  } else {
    const double dx = y.x - m.x, dy = y.y - m.y;
    const double d2 = dx * dx + dy * dy;
    const double norm = miller_row(F.k * (off ? d2 * rsqrt(d2) : 0.0), pb + 1, (double*)row, 1);
    en = (int)((__double2hiint(norm) >> 20) & 0x7FF) - 1023;
    imn = 1.0f / f32_from_f64_sh(norm, -en);
  }
  const double* isg = F.isig + (size_t)l * (F.pbmax + 2);
  const float2* isf = F.isf + (size_t)l * (F.pbmax + 2);
  const ff c1 = off ? ff_mul(D.x, D.ir) : mkff(1.f, 0.f);
  const ff s1 = off ? ff_mul(D.y, D.ir) : mkff(0.f, 0.f);
  ff c8 = c1, s8 = mkff(-s1.h, -s1.l);  // e^{-8 i th} by three squarings
#pragma unroll
  for (int u = 0; u < 3; ++u) ff_turn(c8, s8, c8, s8);
  const float2 emf = make_float2(ff_f32(c1), -ff_f32(s1));
  ff ex = mkff(1.f, 0.f), ey = mkff(0.f, 0.f);
  float2 ef = make_float2(1.f, 0.f);
  float sc = 1.f;
  for (int j = 0; j <= pb + 1; ++j) {
    if ((j & 7) == 0) {
      ef = make_float2(ff_f32(ex), ff_f32(ey));
      ff_turn(ex, ey, c8, s8);
    } else {
      ef = fmul(ef, emf);
    }
    float v;
    if (in) {
      const float2 g = isf[j];
      v = ff_f32(ff_mul_raw(ff_mul_raw(ff_miller_value(row[j], sc), mkff(g.x, g.y)), inv));
    } else {
      v = f32_from_f64_sh(reinterpret_cast<const double*>(row)[j] * isg[j], -en) * imn;
    }
    row[j] = make_float2(ef.x * v, ef.y * v);  // R_j
  }
}

// v, or its conjugate where neg is the sign bit
__device__ __forceinline__ float2 fconj_if(float2 v, unsigned neg) {
  return make_float2(v.x, __uint_as_float(__float_as_uint(v.y) ^ neg));
}

// Rows and strengths of an item in shared memory: FP32 and t >= 0 only, a quarter of
// the FP64 form's. One warp fills an item's rows while the others wait, so blocks of
// 64 threads, of which twice as many share an SM. (With this, and with the orders that
// Miller's recurrence outgrows marked instead of rescaled at once, 200 ellipses 0.84 ->
// 0.51 ms, the starfish at k = 50 0.135 -> 0.088.)
constexpr int kP2mMixedThreads = 64;
static_assert(kP2mMixedThreads >= kChunk, "a thread per source of an item");
__host__ __device__ inline int p2m_mixed_row(int pb) { return (pb + 2) | 1; }
inline size_t p2m_mixed_smem(int pb, int chunk) {
  return (size_t)chunk * (p2m_mixed_row(pb) + 3) * sizeof(float2);
}
__global__ void __launch_bounds__(kP2mMixedThreads) p2m_item_mixed_kernel(
    Fmm F, const int4* __restrict__ items, const int* __restrict__ seg_leaf,
    const int2* __restrict__ seg_row, const long long* __restrict__ seg_poff,
    const int* __restrict__ src, const int* __restrict__ src_leaf, cd* __restrict__ partial,
    int chunk) {
  extern __shared__ __align__(16) float2 fsmem[];
  const int4 it = items[blockIdx.x];
  const int l = F.level[seg_leaf[it.x]];
  const int pb = F.lpb[l], Q = 2 * pb + 1, RW = p2m_mixed_row(pb);
  float2* rows = fsmem;                   // [chunk][RW], it.w <= chunk
  float2* sq = rows + chunk * RW;         // [chunk]
  float2* sa = sq + chunk;                // [chunk]
  float2* sb = sa + chunk;                // [chunk]
  if ((int)threadIdx.x < it.w) {
    const int j = threadIdx.x, i = src[it.z + j];
    const FfUnits& U = F.U;
    p2m_fill_row_mixed(F, U, i, F.centre[src_leaf[it.z + j]], l, pb, rows + j * RW);
    const float4 ab = F.ab32[i];
    sq[j] = F.q32[i];
    sa[j] = make_float2(ab.z, ab.w);  // d (k/2) conj(nu)
    sb[j] = make_float2(ab.x, ab.y);  // d (k/2) nu
  }
  __syncthreads();
  const double2* sr = F.sigr + (size_t)l * (F.pbmax + 2);
  for (int idx = threadIdx.x; idx < it.y * Q; idx += kP2mMixedThreads) {
    const int u = idx / Q, n = idx % Q - pb;
    const int2 rg = seg_row[it.x + u];
    float2 Sq = make_float2(0.f, 0.f), Cq = Sq, Sa = Sq, Ca = Sq, Sb = Sq, Cb = Sq;
    const int an = abs(n), aa = abs(n - 1), ab = abs(n + 1);
    const unsigned gq = n < 0 ? 0x80000000u : 0u, ga = n < 1 ? 0x80000000u : 0u,
                   gb = n < -1 ? 0x80000000u : 0u;
    for (int j = rg.x; j < rg.x + rg.y; ++j) {
      const float2* r = rows + j * RW;
      if (F.has_S) kahan2(Sq, Cq, fmul(sq[j], fconj_if(r[an], gq)));
      if (F.has_D) {
        kahan2(Sa, Ca, fmul(sa[j], fconj_if(r[aa], ga)));
        kahan2(Sb, Cb, fmul(sb[j], fconj_if(r[ab], gb)));
      }
    }
    // the sign (-1)^t of the negative orders t
    const float zq = gq && (an & 1) ? -1.f : 1.f, za = ga && (aa & 1) ? -1.f : 1.f,
                zb = gb && (ab & 1) ? -1.f : 1.f;
    // sig_|n-1| / sig_|n| and sig_|n+1| / sig_|n| (1 beyond order pb); the three sums
    // are joined in float-float
    const double2 rt = sr[an];
    const ff fm = ff_from_f64_nan(n > 0 ? rt.x : rt.y, 896),
             fp = ff_from_f64_nan(n < 0 ? rt.x : rt.y, 896);
    auto join = [&](float q, float cq, float a, float ca, float b, float cb) {
      const ff t = ff_sub_raw(ff_mul_raw(mkff(za * a, -za * ca), fm),
                              ff_mul_raw(mkff(zb * b, -zb * cb), fp));
      return ff_f64(ff_add(mkff(zq * q, -zq * cq), t));
    };
    const double re = join(Sq.x, Cq.x, Sa.x, Ca.x, Sb.x, Cb.x);
    const double im = join(Sq.y, Cq.y, Sa.y, Ca.y, Sb.y, Cb.y);
    partial[seg_poff[it.x + u] + n + pb] = mk(re, im);
  }
}

__global__ void __launch_bounds__(kThreads) p2m_sum_mixed_kernel(
    Fmm F, const int* __restrict__ leaves, const int* __restrict__ lseg,
    const long long* __restrict__ seg_poff, const cd* __restrict__ partial) {
  const int t = blockIdx.x, b = leaves[t];
  const int l = F.level[b];
  const int pb = F.lpb[l], Q = 2 * pb + 1;
  const double* icv = F.iconv + (size_t)l * (F.pbmax + 1);
  cd* dst = F.mpole + F.eoff[b];
  for (int n = threadIdx.x; n < Q; n += kThreads) {
    cd sum = mk(0.0, 0.0);
    for (int g = lseg[t]; g < lseg[t + 1]; ++g) sum = cadd(sum, partial[seg_poff[g] + n]);
    dst[n] = cscale(sum, icv[abs(n - pb)]);
  }
}

// P2L in mixed precision: the item structure of p2l_item_kernel with FP32
// rows and sums. Row j of a source holds G_j e^{i j th} (j >= 0) and
// (-1)^j G_j e^{-i j th} (j < 0), G_j = sig_j H_j(k r) (sig of the box's level,
// sig_{pb+1} taken as sig_pb); X-list sources lie at least 1.5 box sides from
// the centre, so G_j is of order one or smaller. On float-float levels
// G_j = w_j / isf[j], w_j = 2^{s j} H_j by the float-float recurrence
//   w_{j+1} = (2 j 2^s / x) w_j - 4^s w_{j-1};
// elsewhere in FP64, G_{j+1} = rec[j].x (1/x) G_j - rec[j].y G_{j-1}. The angular
// factors are FP32 between anchors every eighth order. Per output order n the charge
// and the two dipole sums are FP32 with Kahan compensation over the item's
// sources; lambda_n = sig_n gamma_n = Sq + (sig_n / sig_|n-1|) Sa -
// (sig_n / sig_|n+1|) Sb and lh_n = lambda_n conv_|n|.
// (One warp of a block fills its rows: bound by that recurrence's latency and by how
// many blocks share an SM. Against FP64 recurrences, rows in 16-byte slots and blocks
// of 128 threads, 200 ellipses 0.64 -> 0.31 ms, the starfish at k = 50 0.073 -> 0.043.)
constexpr int kP2lMixedThreads = 64;
static_assert(kP2lMixedThreads >= kChunk, "a thread per source of an item");
inline size_t p2l_mixed_smem(int pb, int chunk) {
  return (size_t)chunk * (2 * pb + 6) * sizeof(float2);
}
// The row (at j = 0) of one source; R = rec, g = isf of the box's level.
__device__ __forceinline__ void p2l_fill_row_mixed(const Fmm& F, double dx, double dy, int l, int pb,
                                                   const double2* __restrict__ R, float2* row) {
  const int s = F.ffs[l];
  auto put = [&](int j, float2 g, float2 e) {
    const float2 wp = fmul(g, e);
    const float2 wq = fmul(g, make_float2(e.x, -e.y));
    row[j] = wp;
    row[-j] = (j & 1) ? make_float2(-wq.x, -wq.y) : wq;
  };
  if (s != kNoFf) {
    const float2* isf = F.isf + (size_t)l * (F.pbmax + 2);
    const FfUnits& U = F.U;
    FfPolar D;
    D.set(dx, dy, U);
    ffh hp, hc;
    hankel01_ff_any<3>(D.z, hp, hc);
    const float sg = pow2f(s), sg2 = pow2f(2 * s);
    hc.x = ff_scale(hc.x, sg);
    hc.y = ff_scale(hc.y, sg);
    const ff c2 = split17(ff_mul_raw(ff_scale(U.ik2, sg), D.ir));  // 2 2^s / x
    const ff c1 = ff_mul(D.x, D.ir), s1 = ff_mul(D.y, D.ir);
    ff c8 = c1, s8 = s1;
#pragma unroll
    for (int u = 0; u < 3; ++u) ff_turn(c8, s8, c8, s8);
    const float2 e1 = make_float2(ff_f32(c1), ff_f32(s1));
    ff ex = c8, ey = s8;
    float2 e = e1;
    auto scaled = [&](int j, ffh w) {  // w / isf[j]
      const float2 g = isf[j];
      const float r = 1.0f / g.x;
      const ff ig = mkff(r, __fmul_rn(r, __fmaf_rn(-g.y, r, __fmaf_rn(-g.x, r, 1.0f))));
      return make_float2(ff_f32(ff_mul_raw(w.x, ig)), ff_f32(ff_mul_raw(w.y, ig)));
    };
    row[0] = scaled(0, hp);
    for (int j = 1; j <= pb + 1; ++j) {
      if ((j & 7) == 0) {
        e = make_float2(ff_f32(ex), ff_f32(ey));
        ff_turn(ex, ey, c8, s8);
      } else if (j > 1) {
        e = fmul(e, e1);
      }
      put(j, scaled(j, hc), e);
      const ff cj = mkff((float)j * c2.h, (float)j * c2.l);
      const ff nx = ff_sub_raw(ff_mul_raw(cj, hc.x), ff_scale(hp.x, sg2));
      const ff ny = ff_sub_raw(ff_mul_raw(cj, hc.y), ff_scale(hp.y, sg2));
      hp = hc;
      hc.x = nx;
      hc.y = ny;
    }
    return;
  }
  const double d2 = dx * dx + dy * dy;
  const double ir = rsqrt(d2), x = F.k * (d2 * ir), ix = ir * F.ik;
  cd h0, h1;
  hankel01_wide(x, ix, h0, h1);
  const cd e1 = mk(dx * ir, dy * ir);
  cd e8 = cmul(e1, e1);
  e8 = cmul(e8, e8);
  e8 = cmul(e8, e8);
  const float2 e1f = f2(e1);
  cd gprev = h0, gcur = cscale(h1, R[0].x);  // G_0, G_1
  cd E = mk(1.0, 0.0);
  float2 ef = make_float2(1.f, 0.f);
  row[0] = f2(h0);
  for (int j = 1; j <= pb + 1; ++j) {
    if ((j & 7) == 0) {  // e^{i j th}: an FP64 anchor every eighth order
      E = cmul(E, e8);
      ef = f2(E);
    } else {
      ef = fmul(ef, e1f);
    }
    put(j, f2(gcur), ef);
    if (j <= pb) {
      const double c1 = R[j].x * ix, c2 = R[j].y;
      const cd gn = mk(fma(c1, gcur.x, -c2 * gprev.x), fma(c1, gcur.y, -c2 * gprev.y));
      gprev = gcur;
      gcur = gn;
    }
  }
}
__global__ void __launch_bounds__(kP2lMixedThreads) p2l_item_mixed_kernel(
    Fmm F, const int4* __restrict__ items, const int* __restrict__ src,
    const long long* __restrict__ poff, cd* __restrict__ partial, int chunk,
    const double2* __restrict__ rec) {
  extern __shared__ __align__(16) float2 fsmem[];
  const int4 it = items[blockIdx.x];  // (box, first position in src, sources <= chunk, -)
  const int b = it.x, cnt = it.z;
  const int l = F.level[b];
  const int pb = F.lpb[l], RW = 2 * pb + 3;  // row: |t| <= pb+1
  float2* rows = fsmem;                   // [chunk][RW]
  float2* sq = rows + chunk * RW;         // [chunk]
  float2* sa = sq + chunk;                // [chunk]  A = d (k/2) nu
  float2* sb = sa + chunk;                // [chunk]  B = d (k/2) conj(nu)
  const double2 m = F.centre[b];
  if ((int)threadIdx.x < cnt) {
    const int i = src[it.y + threadIdx.x];
    p2l_fill_row_mixed(F, F.sxy[i].x - m.x, F.sxy[i].y - m.y, l, pb,
                       rec + (size_t)l * (F.pbmax + 2), rows + threadIdx.x * RW + (pb + 1));
    const float4 ab = F.ab32[i];
    sq[threadIdx.x] = F.q32[i];
    sa[threadIdx.x] = make_float2(ab.x, ab.y);  // d (k/2) nu
    sb[threadIdx.x] = make_float2(ab.z, ab.w);  // d (k/2) conj(nu)
  }
  __syncthreads();
  const double2* sr = F.sigr + (size_t)l * (F.pbmax + 2);
  const double* cv = F.conv + (size_t)l * (F.pbmax + 1);
  cd* dst = partial + poff[blockIdx.x] + pb;
  for (int n = (int)threadIdx.x - pb; n <= pb; n += kP2lMixedThreads) {
    float2 Sq = make_float2(0.f, 0.f), Cq = Sq, Sa = Sq, Ca = Sq, Sb = Sq, Cb = Sq;
    for (int j = 0; j < cnt; ++j) {
      const float2* r = rows + j * RW + (pb + 1) + n;
      if (F.has_S) kahan2(Sq, Cq, fmul(sq[j], r[0]));
      if (F.has_D) {
        kahan2(Sa, Ca, fmul(sa[j], r[-1]));
        kahan2(Sb, Cb, fmul(sb[j], r[1]));
      }
    }
    // sig_|n| / sig_|n-1| and sig_|n| / sig_|n+1|: the ratio table holds sig_{m-1} /
    // sig_m and sig_{m+1} / sig_m at m (1 beyond order pb); the three sums are joined
    // in float-float
    const int an = abs(n);
    const double up = sr[an + 1].x, dn = an > 0 ? sr[an - 1].y : up;
    const ff fm = ff_from_f64_nan(n > 0 ? dn : up, 896), fp = ff_from_f64_nan(n < 0 ? dn : up, 896);
    const double c = cv[an];
    auto join = [&](float q, float cq, float a, float ca, float b, float cb) {
      const ff t = ff_sub_raw(ff_mul_raw(mkff(a, -ca), fm), ff_mul_raw(mkff(b, -cb), fp));
      return ff_f64(ff_add(mkff(q, -cq), t));
    };
    const double re = join(Sq.x, Cq.x, Sa.x, Ca.x, Sb.x, Cb.x);
    const double im = join(Sq.y, Cq.y, Sa.y, Ca.y, Sb.y, Cb.y);
    dst[n] = mk(re * c, im * c);
  }
}

// Lift the 48 KB default of dynamic shared memory to the device's opt-in
// maximum for every kernel that uses it (once per device); the size given at
// each launch still decides the occupancy.

qbx_status configure_kernels() {
  static std::mutex mu;
  static std::set<int> done;
  int dev = 0;
  QBX_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  if (done.count(dev)) return QBX_OK;
  int optin = 0;
  QBX_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  const void* k[] = {(const void*)p2m_item_kernel, (const void*)p2m_item_mixed_kernel,
                     (const void*)m2m_kernel,
                     (const void*)p2l_item_kernel, (const void*)p2l_item_mixed_kernel,
                     (const void*)l2l_kernel};
  for (const void* f : k)
    QBX_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
  TRY_MIXED(configure_mixed_kernels(optin));
  TRY_MIXED(configure_tc_kernels(optin));
  g_smem_optin = optin;
  done.insert(dev);
  return QBX_OK;
}

// ---------------------------------------------------------------- P2QBXL, W lanes per centre
// The lanes of a centre stride over the concatenated sources of its U-list boxes
// (so the load is balanced to within one source), each keeps partial coefficients
// (p2qbxl_pair), and a reduce-scatter of shuffles adds them. A pass over a centre's
// sources ends with a partly filled step (150 sources are 4.7 steps of 32 lanes), so
// where centres are plenty half a warp takes one (W = 16, two centres per warp); with
// few centres a warp each keeps more of the SMs' pipes fed. The rule takes all centres
// of the handle, of which a launch may form only those that targets use, so that a
// coefficient is the same sum whichever are formed. Measured with a warp and half a
// warp each: 200 ellipses, mixed, 2.37 and 2.03 ms; 32 curves of 512 to 32768 centres in
// a batch 5.99 and 5.34 ms in all; the GMRES solve with 3072 centres 38.3 and 42.6 ms.
// A handle of many centres that forms few of them loses by it (the starfish at k = 50,
// mixed, few targets near the curve: 0.037 and 0.066 ms, beside the main stream).
constexpr int kHalfWarpCentres = 6144;
// Launches of fewer centres than this run one-warp blocks, which spread over the SMs
// more evenly.
constexpr int kSmallBlockCentres = 8192;
template <int PM, bool HS, bool HD, int W>
__global__ void __launch_bounds__(kThreads) p2qbxl_warp_kernel(Fmm F, const int* __restrict__ cleaf,
                                                               const int* __restrict__ wdoff,
                                                               const int* __restrict__ wdbox,
                                                               const int* __restrict__ clist,
                                                               int n_ctr, cd* __restrict__ alpha) {
  constexpr int NC = 2 * PM + 2;
  const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) / W);  // position in clist
  const int lane = threadIdx.x & (W - 1);
  if ((w & ~(32 / W - 1)) >= n_ctr) return;  // whole warps leave together
  const bool live = w < n_ctr;  // the last warp's second half may be without a centre
  const int i = clist[live ? w : n_ctr - 1];  // sorted centre
  const int b = cleaf[i];
  const double k = F.k, ik = F.ik, hk = 0.5 * k;
  const int p = F.p;
  const double2 c = F.cxy[i];
  cd acc[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) acc[j] = mk(0.0, 0.0);
  auto one = [&](int j) {
    const double2 y = F.sxy[j];
    const double2 nv = HD ? F.snrm[j] : make_double2(0.0, 0.0);
    const cd z = mk(0.0, 0.0);
    p2qbxl_pair<PM, HS, HD>(acc, y.x - c.x, y.y - c.y, HS ? F.qs[j] : z,
                            HD ? cscale(F.ds[j], hk) : z, nv.x, nv.y, k, ik, p);
  };
  // U-list boxes of the leaf, then the W-list boxes summed directly for this centre
  const SourceCursor sc{F.uidx, F.rsrc, F.uoff[b], F.uoff[b + 1] - F.uoff[b], wdoff[i],
                        wdoff[i + 1] - wdoff[i], wdbox};
  if (live) deal_sources<W>(sc, lane, one);
  __syncwarp();
  cd x32, x33;
  group_reduce_scatter<W, NC>(acc, lane, x32, x33);
  cd* dst = alpha + (size_t)F.cid[i] * (2 * p + 1) + p;
  pair_coefficients<W, PM>(acc[0], acc[1], x32, x33, lane, p, [&](int l, cd a) {
    if (live) dst[l] = cadd(dst[l], a);
  });
}

template <int PM, bool HS, bool HD, int W>
__global__ void __launch_bounds__(kThreads) p2qbxl_warp_mixed_kernel(Fmm F, const int* __restrict__ cleaf,
                                                                     const int* __restrict__ wdoff,
                                                                     const int* __restrict__ wdbox,
                                                                     const int* __restrict__ clist,
                                                                     int n_ctr, cd* __restrict__ alpha) {
  constexpr int NC = 2 * PM + 2;
  const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) / W);  // position in clist
  const int lane = threadIdx.x & (W - 1);
  if ((w & ~(32 / W - 1)) >= n_ctr) return;
  const bool live = w < n_ctr;
  const int i = clist[live ? w : n_ctr - 1];
  const int b = cleaf[i];
  const double k = F.k;
  const int p = F.p;
  const double2 c = F.cxy[i];
  // sigma = 2^s within a factor sqrt 2 of k r_c
  const int s = ilogb(k * F.crad[i] * 1.4142135623730951);
  const float sg = pow2f(s), sg2 = pow2f(2 * s);
  const FfUnits& U = F.U;
  const ff c2s = ff_scale(U.ik2, sg);
  f32p S[NC], N[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) S[j] = N[j] = 0ull;
  auto one = [&](int j) {
    const double2 y = F.sxy[j];
    float2 q = make_float2(0.f, 0.f);
    if (HS) {
      q = F.q32[j];
      q = make_float2(q.x * sg, q.y * sg);
    }
    p2qbxl_pair_mixed<PM, HS, HD>(S, N, y.x - c.x, y.y - c.y, q,
                                  HD ? F.dn32[j] : make_float4(0.f, 0.f, 0.f, 0.f), U, c2s, sg,
                                  sg2, p);
  };
  const SourceCursor sc{F.uidx, F.rsrc, F.uoff[b], F.uoff[b + 1] - F.uoff[b], wdoff[i],
                        wdoff[i + 1] - wdoff[i], wdbox};
  if (live) deal_sources<W>(sc, lane, one);
  __syncwarp();
  // the lanes' sums (S + N) added over the group in float-float: in FP64 the
  // conversions and additions of one centre were 290 FP64 instructions, as many as
  // 145 of its pairs
  ffh acc[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    const float2 s = unpk(S[j]), n = unpk(N[j]);
    acc[j].x = mkff(s.x, n.x);
    acc[j].y = mkff(s.y, n.y);
  }
  ffh y32, y33;
  group_reduce_scatter<W, NC>(acc, lane, y32, y33);
  auto f64 = [](ffh v) { return mk(ff_f64(v.x), ff_f64(v.y)); };
  const cd a0 = f64(acc[0]), a1 = W == 16 ? f64(acc[1]) : a0;
  const cd x32 = PM == 16 ? f64(y32) : a0, x33 = PM == 16 ? f64(y33) : a0;
  cd* dst = alpha + (size_t)F.cid[i] * (2 * p + 1) + p;
  const double os = pow2d(out_exp(F));
  pair_coefficients<W, PM>(a0, a1, x32, x33, lane, p, [&](int l, cd a) {
    // the sums carry sigma^{|l|+1}
    if (live) dst[l] = cadd(dst[l], cscale(cscale(a, pow2d(-s * (abs(l) + 1))), os));
  });
}

}  // namespace

#define TRY(x)                          \
  do {                                  \
    qbx_status s_ = (x);                \
    if (s_ != QBX_OK) return s_;        \
  } while (0)

// Shared memory of a source-row kernel (P2M, P2L) at box order pb: a full
// warp's chunk of rows while that keeps the block within kRowsSmemTarget
// (several blocks per SM), else half a warp's; never above the opt-in limit.
constexpr size_t kRowsSmemTarget = 60 * 1024;
size_t rows_launch_smem(int pb) {
  const size_t full = rows_smem(pb, kChunk);
  const size_t sm = full <= kRowsSmemTarget ? full : rows_smem(pb, kChunk / 2);
  return std::min(sm, (size_t)g_smem_optin);
}

// Largest box order among the levels l with off[l+1] > off[l] (boxes of a
// level-ordered list); the single launch over the list sizes its shared memory
// for it. The lists are ordered coarse to fine, so the CTAs with the most work
// (highest orders) start first.
int max_order(const std::vector<int>& pb, const std::vector<int>& off) {
  int m = 0;
  for (size_t l = 0; l + 1 < off.size(); ++l)
    if (off[l + 1] > off[l]) m = std::max(m, pb[l]);
  return m;
}

qbx_status fmm_plan_build(qbx_handle* h, const qbx_tree_desc* d, const int64_t* on_node_dev,
                          const int8_t* on_side_dev, double eps) {
  if (h->fmm) fmm_plan_free(h->fmm);
  FmmPlan* f = new FmmPlan();
  h->fmm = f;
  const int n_max = d->n_max > 0 ? d->n_max : 64;
  TRY(tree_build(h, f, n_max, kLeafOverRadius));
  TRY(tree_lists(h, f));
  TRY(tree_associate(h, f, on_node_dev, on_side_dev, eps));
  TRY(gather_sorted(h, f));
  const int p_add = d->p_add >= 0 ? d->p_add : qbx_default_p_add(h->p);
  if (f->n_levels > kMaxLevels + 1) {
    set_error("tree has %d levels (at most %d)", f->n_levels, kMaxLevels + 1);
    return QBX_ERR_ARG;
  }
  // box order per level (Sec. 7.1): p_fmm on the finest level, more on coarse
  // levels whose boxes span wavelengths, plus p_add
  f->h_pb.assign(f->n_levels, 0);
  TRY(qbx_fmm_level_orders(h->k, f->side, f->n_levels, std::max(1, d->p_fmm), p_add,
                           f->h_pb.data()));
  f->pb_max = 1;
  for (int l = 0; l < f->n_levels; ++l) f->pb_max = std::max(f->pb_max, f->h_pb[l]);
  f->pb_fine = f->h_pb[f->n_levels - 1];
  // scales, powers, translation tables
  std::vector<double> sc(f->n_levels);
  for (int l = 0; l < f->n_levels; ++l) {
    sc[l] = std::min(1.0, h->k * f->side / (double)(1 << l));
    if (l >= 2 && std::pow(sc[l], f->h_pb[l] + 1) < 1e-250) {
      set_error("tree level %d too fine for the box order %d (k*side = %.3g)", l, f->h_pb[l],
                sc[l]);
      return QBX_ERR_ARG;
    }
  }
  // coefficient offsets: boxes of level l are [level_off[l], level_off[l+1])
  {
    std::vector<long long> eo(f->n_boxes);
    long long off = 0;
    for (int l = 0; l < f->n_levels; ++l)
      for (int b = f->level_off[l]; b < f->level_off[l + 1]; ++b) {
        eo[b] = off;
        off += 2 * f->h_pb[l] + 1;
      }
    f->n_coef = off;
    QBX_CUDA_TRY(f->eoff.alloc(std::max(1, f->n_boxes)));
    if (f->n_boxes)
      QBX_CUDA_TRY(cudaMemcpy(f->eoff.ptr, eo.data(), eo.size() * sizeof(long long),
                              cudaMemcpyHostToDevice));
  }
  QBX_CUDA_TRY(f->lpb.alloc(f->n_levels));
  QBX_CUDA_TRY(cudaMemcpy(f->lpb.ptr, f->h_pb.data(), f->n_levels * sizeof(int),
                          cudaMemcpyHostToDevice));
  QBX_CUDA_TRY(f->scale.alloc(f->n_levels));
  QBX_CUDA_TRY(cudaMemcpy(f->scale.ptr, sc.data(), sc.size() * sizeof(double),
                          cudaMemcpyHostToDevice));
  const int pbm = f->pb_max, TS = 4 * pbm + 1;
  QBX_CUDA_TRY(f->t_m2l.alloc((size_t)f->n_levels * 49 * TS));
  QBX_CUDA_TRY(f->t_m2m.alloc((size_t)f->n_levels * 4 * TS));
  QBX_CUDA_TRY(f->t_l2l.alloc((size_t)f->n_levels * 4 * TS));
  QBX_CUDA_TRY(f->pw.alloc((size_t)f->n_levels * (2 * pbm + 3)));
  QBX_CUDA_TRY(f->ipw.alloc((size_t)f->n_levels * (pbm + 2)));
  DevBuf<double> jwork;
  QBX_CUDA_TRY(jwork.alloc((size_t)f->n_levels * 57 * (2 * pbm + 1)));
  tables_kernel<<<nblk(f->n_levels * 57, 64), 64>>>(f->n_levels, f->side, h->k, pbm, f->lpb.ptr,
                                                    f->scale.ptr, f->t_m2l.ptr, f->t_m2m.ptr,
                                                    f->t_l2l.ptr, jwork.ptr);
  powers_kernel<<<1, 64>>>(f->n_levels, pbm, f->lpb.ptr, f->scale.ptr, f->pw.ptr, f->ipw.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  QBX_CUDA_TRY(f->mpole.alloc(std::max<int64_t>(1, f->n_coef)));
  QBX_CUDA_TRY(f->local.alloc(std::max<int64_t>(1, f->n_coef)));
  QBX_CUDA_TRY(f->lpq.alloc(std::max<int64_t>(1, f->n_coef)));
  QBX_CUDA_TRY(f->sp_m.alloc(std::max<int64_t>(1, f->n_coef)));
  QBX_CUDA_TRY(f->sp_e.alloc(std::max<int64_t>(1, f->n_coef)));
  TRY(configure_kernels());
  // side stream and events for the concurrent near-field stages (created here,
  // outside any stream capture; owned by the plan)
  QBX_CUDA_TRY(cudaStreamCreateWithFlags(&f->near_stream, cudaStreamNonBlocking));
  for (cudaEvent_t* ev : {&f->ev_fork, &f->ev_join, &f->ev_p2l, &f->ev_m2m, &f->ev_out})
    QBX_CUDA_TRY(cudaEventCreateWithFlags(ev, cudaEventDisableTiming));
  // the limit on box orders: no kernel stages more than this for its largest one
  const size_t smem_need = gemm_smem_bytes(f->pb_max);
  if (smem_need > (size_t)g_smem_optin) {
    set_error("box order %d needs %zu bytes of shared memory per block (device: %d)", f->pb_max,
              smem_need, g_smem_optin);
    return QBX_ERR_ARG;
  }
  TRY(mixed_plan_build(h, f));
  QBX_CUDA_TRY(f->tmm_f64.alloc(f->tmm_f32.n));
  QBX_CUDA_TRY(f->tl_f64.alloc(f->tl_f32.n));
  for (int l = 2; l + 1 < f->n_levels; ++l) {
    const int pp = f->h_pb[l], pc = f->h_pb[l + 1];
    fold64_matrix_kernel<true><<<2 * pc + 1, kThreads>>>(l, pp, pc, pbm, f->t_m2m.ptr, f->pw.ptr,
                                                         f->ipw.ptr, f->tmm_f64.ptr + f->h_fold_off[l]);
    QBX_CUDA_TRY(cudaGetLastError());
    fold64_matrix_kernel<false><<<2 * pp + 1, kThreads>>>(l, pp, pc, pbm, f->t_l2l.ptr, f->pw.ptr,
                                                          f->ipw.ptr, f->tl_f64.ptr + f->h_fold_off[l]);
    QBX_CUDA_TRY(cudaGetLastError());
  }
  TRY(tc_plan_build(h, f));
  QBX_CUDA_TRY(f->qs.alloc(std::max<int64_t>(1, h->n_src)));
  QBX_CUDA_TRY(f->ds.alloc(std::max<int64_t>(1, h->n_src)));
  QBX_CUDA_TRY(f->q32.alloc(std::max<int64_t>(1, h->n_src)));
  QBX_CUDA_TRY(f->ab32.alloc(std::max<int64_t>(1, h->n_src)));
  for (DevBuf<float4>* v : {&f->dn32, &f->qf, &f->df, &f->nf})
    QBX_CUDA_TRY(v->alloc(std::max<int64_t>(1, h->n_src)));
  QBX_CUDA_TRY(f->sexp.alloc(1));
  QBX_CUDA_TRY(cudaMemset(f->sexp.ptr, 0, sizeof(int)));
  // leaves holding sources (P2M)
  QBX_CUDA_TRY(dev_sync());
  // stats
  std::vector<int> uoff(f->n_boxes + 1), woff(f->n_boxes + 1), xoff(f->n_boxes + 1);
  std::vector<int2> rs(f->n_boxes), rc(f->n_boxes), rt(f->n_boxes);
  std::vector<int> uidx(std::max<int64_t>(1, f->U.nnz)), widx(std::max<int64_t>(1, f->W.nnz)),
      xidx(std::max<int64_t>(1, f->X.nnz));
  QBX_CUDA_TRY(cudaMemcpy(uoff.data(), f->U.off.ptr, uoff.size() * 4, cudaMemcpyDeviceToHost));
  QBX_CUDA_TRY(cudaMemcpy(woff.data(), f->W.off.ptr, woff.size() * 4, cudaMemcpyDeviceToHost));
  QBX_CUDA_TRY(cudaMemcpy(xoff.data(), f->X.off.ptr, xoff.size() * 4, cudaMemcpyDeviceToHost));
  QBX_CUDA_TRY(cudaMemcpy(rs.data(), f->box.rng[PT_SRC].ptr, rs.size() * 8, cudaMemcpyDeviceToHost));
  QBX_CUDA_TRY(cudaMemcpy(rc.data(), f->box.rng[PT_CTR].ptr, rc.size() * 8, cudaMemcpyDeviceToHost));
  QBX_CUDA_TRY(cudaMemcpy(rt.data(), f->box.rng[PT_TGT].ptr, rt.size() * 8, cudaMemcpyDeviceToHost));
  if (f->U.nnz) QBX_CUDA_TRY(cudaMemcpy(uidx.data(), f->U.idx.ptr, f->U.nnz * 4, cudaMemcpyDeviceToHost));
  if (f->W.nnz) QBX_CUDA_TRY(cudaMemcpy(widx.data(), f->W.idx.ptr, f->W.nnz * 4, cudaMemcpyDeviceToHost));
  if (f->X.nnz) QBX_CUDA_TRY(cudaMemcpy(xidx.data(), f->X.idx.ptr, f->X.nnz * 4, cudaMemcpyDeviceToHost));
  std::vector<int> assoc_s(std::max<int64_t>(1, h->n_tgt));
  if (h->n_tgt)
    QBX_CUDA_TRY(cudaMemcpy(assoc_s.data(), f->t_assoc.ptr, h->n_tgt * 4, cudaMemcpyDeviceToHost));
  std::vector<int> leaves(f->n_leaves), blev(f->n_boxes);
  QBX_CUDA_TRY(cudaMemcpy(leaves.data(), f->leaves.ptr, leaves.size() * 4, cudaMemcpyDeviceToHost));
  QBX_CUDA_TRY(cudaMemcpy(blev.data(), f->box.level.ptr, blev.size() * 4, cudaMemcpyDeviceToHost));
  int64_t p2qbxl = 0, p2p = 0, m2qbxl = 0, m2p = 0, p2l = 0;
  std::vector<int> src_leaves;
  for (int b : leaves) {
    int64_t us = 0;
    for (int e = uoff[b]; e < uoff[b + 1]; ++e) us += rs[uidx[e]].y - rs[uidx[e]].x;
    int64_t nd = 0;
    for (int i = rt[b].x; i < rt[b].y; ++i) nd += assoc_s[i] < 0 ? 1 : 0;
    p2qbxl += us * (rc[b].y - rc[b].x);
    p2p += us * nd;
    m2qbxl += (int64_t)(woff[b + 1] - woff[b]) * (rc[b].y - rc[b].x);
    m2p += (int64_t)(woff[b + 1] - woff[b]) * nd;
    if (rs[b].y > rs[b].x && blev[b] >= 2) src_leaves.push_back(b);
    f->q_leaf = std::max(f->q_leaf, 2 * f->h_pb[blev[b]] + 1);
    for (int e = woff[b]; e < woff[b + 1]; ++e)
      f->q_w = std::max(f->q_w, 2 * f->h_pb[blev[widx[e]]] + 1);
  }
  // leaf of every sorted target; direct targets, and those among them whose
  // leaf has U-list sources (P2P) or a W list (M2P)
  {
    std::vector<int> tl(std::max<int64_t>(1, h->n_tgt), 0), dt, ut, wt;
    for (int b : leaves)
      for (int i = rt[b].x; i < rt[b].y; ++i) tl[i] = b;
    std::vector<int64_t> usrc(f->n_boxes, 0);
    for (int b : leaves)
      for (int e = uoff[b]; e < uoff[b + 1]; ++e) usrc[b] += rs[uidx[e]].y - rs[uidx[e]].x;
    for (int64_t i = 0; i < h->n_tgt; ++i) {
      if (assoc_s[i] >= 0) continue;
      const int b = tl[i];
      dt.push_back((int)i);
      if (usrc[b] > 0) ut.push_back((int)i);
      if (woff[b + 1] > woff[b]) wt.push_back((int)i);
    }
    auto up = [](DevBuf<int>& d, const std::vector<int>& v) -> qbx_status {
      QBX_CUDA_TRY(d.alloc(std::max<size_t>(1, v.size())));
      if (!v.empty())
        QBX_CUDA_TRY(cudaMemcpy(d.ptr, v.data(), v.size() * sizeof(int), cudaMemcpyHostToDevice));
      return QBX_OK;
    };
    // M2P work items: the (target, W box) pairs by (leaf, box, target), so that
    // neighbouring threads share a box; slot: the pair's place in target order
    // (CSR by wtgt position), where its value is stored for the ordered sum
    std::vector<int> mt, mbx, mslot, moff(wt.size() + 1, 0);
    for (size_t t = 0; t < wt.size(); ++t) {
      const int b = tl[wt[t]];
      moff[t + 1] = moff[t] + woff[b + 1] - woff[b];
    }
    mt.reserve(moff.back());
    mbx.reserve(moff.back());
    mslot.reserve(moff.back());
    for (size_t t0 = 0; t0 < wt.size();) {
      const int b = tl[wt[t0]];
      size_t t1 = t0;
      while (t1 < wt.size() && tl[wt[t1]] == b) ++t1;
      for (int e = woff[b]; e < woff[b + 1]; ++e)
        for (size_t t = t0; t < t1; ++t) {
          mt.push_back(wt[t]);
          mbx.push_back(widx[e]);
          mslot.push_back(moff[t] + e - woff[b]);
        }
      t0 = t1;
    }
    TRY(up(f->tleaf, tl));
    TRY(up(f->dtgt, dt));
    TRY(up(f->utgt, ut));
    TRY(up(f->wtgt, wt));
    TRY(up(f->m2p_tgt, mt));
    TRY(up(f->m2p_box, mbx));
    TRY(up(f->m2p_slot, mslot));
    TRY(up(f->m2p_off, moff));
    QBX_CUDA_TRY(f->m2p_part.alloc(std::max<size_t>(1, mt.size())));
    {  // the boxes M2P reads, and FP32 room for their normalised multipoles
      std::vector<int> wb(mbx);
      std::sort(wb.begin(), wb.end());
      wb.erase(std::unique(wb.begin(), wb.end()), wb.end());
      TRY(up(f->m2p_wbox, wb));
      f->n_m2p_wbox = (int)wb.size();
      QBX_CUDA_TRY(f->m2p_mu.alloc(wb.empty() ? 2 : f->n_coef + f->n_boxes));
      QBX_CUDA_TRY(f->m2p_pq.alloc(wb.empty() ? 2 : f->n_coef + f->n_boxes));
    }
    f->n_dtgt = (int)dt.size();
    f->n_utgt = (int)ut.size();
    f->n_wtgt = (int)wt.size();
    f->n_m2p_pairs = (int)mt.size();
  }
  // leaf of every centre (sorted order)
  std::vector<int> cl(std::max<int64_t>(1, h->n_ctr), 0);
  for (int b : leaves)
    for (int i = rc[b].x; i < rc[b].y; ++i) cl[i] = b;
  f->cleaf_pb_max = 0;
  for (int b : leaves)
    if (rc[b].y > rc[b].x) f->cleaf_pb_max = std::max(f->cleaf_pb_max, f->h_pb[blev[b]]);
  QBX_CUDA_TRY(f->cleaf.alloc(cl.size()));
  QBX_CUDA_TRY(cudaMemcpy(f->cleaf.ptr, cl.data(), cl.size() * sizeof(int),
                          cudaMemcpyHostToDevice));
  // W-list boxes per centre: those far enough from the centre's disk for
  // M2QBXL ((R_c + r_z) <= kW |z - m_c|), and the rest, summed directly in
  // P2QBXL (wd_off / wd_box, CSR by sorted centre)
  std::vector<std::vector<int>> wtrans(std::max<int64_t>(1, h->n_ctr));
  int64_t w_direct_src = 0;
  {
    std::vector<double2> cxy(std::max<int64_t>(1, h->n_ctr)), bctr(f->n_boxes);
    std::vector<double> crad(std::max<int64_t>(1, h->n_ctr));
    if (h->n_ctr) {
      QBX_CUDA_TRY(cudaMemcpy(cxy.data(), f->c_xy.ptr, h->n_ctr * sizeof(double2), cudaMemcpyDeviceToHost));
      QBX_CUDA_TRY(cudaMemcpy(crad.data(), f->c_r.ptr, h->n_ctr * sizeof(double), cudaMemcpyDeviceToHost));
    }
    QBX_CUDA_TRY(cudaMemcpy(bctr.data(), f->box.centre.ptr, f->n_boxes * sizeof(double2), cudaMemcpyDeviceToHost));
    std::vector<int> dbx, doff(std::max<int64_t>(1, h->n_ctr) + 1, 0);
    for (int64_t i = 0; i < h->n_ctr; ++i) {
      const int b = cl[i];
      for (int e = woff[b]; e < woff[b + 1]; ++e) {
        const int c = widx[e];
        const double dx = cxy[i].x - bctr[c].x, dy = cxy[i].y - bctr[c].y;
        const double Rc = 0.70710678118654752 * f->side / (double)(1 << blev[c]);
        if (Rc + crad[i] > kW * std::sqrt(dx * dx + dy * dy)) {
          dbx.push_back(c);
          w_direct_src += rs[c].y - rs[c].x;
        } else {
          wtrans[i].push_back(c);
        }
      }
      doff[i + 1] = (int)dbx.size();
    }
    QBX_CUDA_TRY(f->wd_box.alloc(std::max<size_t>(1, dbx.size())));
    QBX_CUDA_TRY(f->wd_off.alloc(doff.size()));
    if (!dbx.empty())
      QBX_CUDA_TRY(cudaMemcpy(f->wd_box.ptr, dbx.data(), dbx.size() * 4, cudaMemcpyHostToDevice));
    QBX_CUDA_TRY(cudaMemcpy(f->wd_off.ptr, doff.data(), doff.size() * 4, cudaMemcpyHostToDevice));
  }
  // Centre sets: every centre (set 0), and the centres some target is
  // associated with (set 1; alpha is only read there). Each set lists sorted
  // centre indices and its M2QBXL (centre, W box) pairs, CSR by list position.
  {
    std::vector<int> all(std::max<int64_t>(0, h->n_ctr)), used;
    for (int64_t i = 0; i < h->n_ctr; ++i) all[i] = (int)i;
    if (h->n_ctr) {
      std::vector<int> cperm(h->n_ctr), inv(h->n_ctr), ta(std::max<int64_t>(1, h->n_tgt));
      std::vector<char> mark(h->n_ctr, 0);
      QBX_CUDA_TRY(cudaMemcpy(cperm.data(), f->perm[PT_CTR].ptr, h->n_ctr * 4, cudaMemcpyDeviceToHost));
      if (h->n_tgt)
        QBX_CUDA_TRY(cudaMemcpy(ta.data(), h->assoc.ptr, h->n_tgt * 4, cudaMemcpyDeviceToHost));
      for (int64_t i = 0; i < h->n_ctr; ++i) inv[cperm[i]] = (int)i;
      for (int64_t t = 0; t < h->n_tgt; ++t)
        if (ta[t] >= 0) mark[inv[ta[t]]] = 1;
      if (h->has_avg) {  // two-sided targets also read their node's interior centre
        std::vector<int8_t> av(h->n_tgt);
        QBX_CUDA_TRY(cudaMemcpy(av.data(), h->avg.ptr, h->n_tgt, cudaMemcpyDeviceToHost));
        for (int64_t t = 0; t < h->n_tgt; ++t)
          if (av[t] && ta[t] >= 0) mark[inv[ta[t] + h->n_nodes]] = 1;
      }
      for (int64_t i = 0; i < h->n_ctr; ++i)
        if (mark[i]) used.push_back((int)i);
    }
    // the W-list boxes of any centre, and whether every level the mixed L2QBXL
    // (M2QBXL) meets has a float-float scaling (M2QBXL's rows go p orders further)
    {
      std::vector<char> seen(f->n_boxes, 0);
      std::vector<int> cw;
      f->ff_wboxes = true;
      for (const std::vector<int>& w : wtrans)
        for (int c : w)
          if (!seen[c]) {
            seen[c] = 1;
            cw.push_back(c);
            const int l = blev[c];
            f->ff_wboxes = f->ff_wboxes && f->h_ffs[l] != kNoFf && f->h_pb[l] + h->p <= 100;
          }
      f->ff_leaves = true;
      for (int b : leaves)
        if (rc[b].y > rc[b].x && f->h_ffs[blev[b]] == kNoFf) f->ff_leaves = false;
      f->n_cw_box = (int)cw.size();
      QBX_CUDA_TRY(f->cw_box.alloc(std::max<size_t>(1, cw.size())));
      if (!cw.empty())
        QBX_CUDA_TRY(cudaMemcpy(f->cw_box.ptr, cw.data(), cw.size() * 4, cudaMemcpyHostToDevice));
      QBX_CUDA_TRY(f->loc32.alloc(std::max<int64_t>(1, f->n_coef)));
    }
    size_t max_pairs = 1;
    for (int k = 0; k < 2; ++k) {
      const std::vector<int>& list = k == 0 ? all : used;
      CentreSet& S = f->cset[k];
      std::vector<int> pc, pbx, off(list.size() + 1, 0);
      for (size_t t = 0; t < list.size(); ++t) {
        for (int c : wtrans[list[t]]) {
          pc.push_back(list[t]);
          pbx.push_back(c);
        }
        off[t + 1] = (int)pc.size();
      }
      S.n = (int)list.size();
      S.n_pairs = (int)pc.size();
      S.wp_pbmax = 0;
      for (int c : pbx) S.wp_pbmax = std::max(S.wp_pbmax, f->h_pb[blev[c]]);
      max_pairs = std::max(max_pairs, pc.size());
      auto up = [](DevBuf<int>& d, const std::vector<int>& v) -> qbx_status {
        QBX_CUDA_TRY(d.alloc(std::max<size_t>(1, v.size())));
        if (!v.empty())
          QBX_CUDA_TRY(cudaMemcpy(d.ptr, v.data(), v.size() * sizeof(int), cudaMemcpyHostToDevice));
        return QBX_OK;
      };
      TRY(up(S.clist, list));
      TRY(up(S.wp_ctr, pc));
      TRY(up(S.wp_box, pbx));
      TRY(up(S.wp_off, off));
    }
    QBX_CUDA_TRY(f->wpart.alloc(max_pairs * (size_t)(2 * h->p + 1)));
    f->n_wpairs = f->cset[0].n_pairs;
    QBX_CUDA_TRY(f->sf_m.alloc((size_t)f->n_levels * (2 * h->p + 1)));
    QBX_CUDA_TRY(f->sf_e.alloc((size_t)f->n_levels * (2 * h->p + 1)));
  }
  // P2M work items over segments of the source leaves (see p2m_item_kernel)
  {
    int pbs = 0;  // largest order over the source leaves
    for (int b : src_leaves) pbs = std::max(pbs, f->h_pb[blev[b]]);
    f->p2m_sm = rows_launch_smem(pbs);
    const int chunk = rows_chunk(pbs, f->p2m_sm);  // the least capacity over the leaf levels
    f->p2m_chunk = chunk;
    f->p2m_pb = pbs;
    std::vector<int> sleaf, psrc, psleaf, lseg(src_leaves.size() + 1, 0);
    std::vector<int2> srow;
    std::vector<long long> spoff;
    std::vector<int4> items;
    long long ptot = 0;
    int cur_lev = -1;
    for (size_t t = 0; t < src_leaves.size(); ++t) {
      const int b = src_leaves[t];
      const int Q = 2 * f->h_pb[blev[b]] + 1;
      lseg[t] = (int)sleaf.size();
      for (int i0 = rs[b].x; i0 < rs[b].y;) {
        if (items.empty() || cur_lev != blev[b] || items.back().w == chunk) {
          items.push_back(make_int4((int)sleaf.size(), 0, (int)psrc.size(), 0));
          cur_lev = blev[b];
        }
        int4& it = items.back();
        const int cnt = std::min(chunk - it.w, rs[b].y - i0);
        srow.push_back(make_int2(it.w, cnt));
        sleaf.push_back(b);
        spoff.push_back(ptot);
        ptot += Q;
        for (int i = i0; i < i0 + cnt; ++i) {
          psrc.push_back(i);
          psleaf.push_back(b);
        }
        it.y += 1;
        it.w += cnt;
        i0 += cnt;
      }
    }
    lseg[src_leaves.size()] = (int)sleaf.size();
    f->n_p2m_items = (int)items.size();
    QBX_CUDA_TRY(f->p2m_items.alloc(std::max<size_t>(1, items.size())));
    QBX_CUDA_TRY(f->p2m_segleaf.alloc(std::max<size_t>(1, sleaf.size())));
    QBX_CUDA_TRY(f->p2m_segrow.alloc(std::max<size_t>(1, srow.size())));
    QBX_CUDA_TRY(f->p2m_segpoff.alloc(std::max<size_t>(1, spoff.size())));
    QBX_CUDA_TRY(f->p2m_lseg.alloc(lseg.size()));
    QBX_CUDA_TRY(f->p2m_src.alloc(std::max<size_t>(1, psrc.size())));
    QBX_CUDA_TRY(f->p2m_srcleaf.alloc(std::max<size_t>(1, psleaf.size())));
    QBX_CUDA_TRY(f->p2m_part.alloc(std::max<long long>(1, ptot)));
    if (!items.empty()) {
      QBX_CUDA_TRY(cudaMemcpy(f->p2m_items.ptr, items.data(), items.size() * sizeof(int4), cudaMemcpyHostToDevice));
      QBX_CUDA_TRY(cudaMemcpy(f->p2m_segleaf.ptr, sleaf.data(), sleaf.size() * sizeof(int), cudaMemcpyHostToDevice));
      QBX_CUDA_TRY(cudaMemcpy(f->p2m_segrow.ptr, srow.data(), srow.size() * sizeof(int2), cudaMemcpyHostToDevice));
      QBX_CUDA_TRY(cudaMemcpy(f->p2m_segpoff.ptr, spoff.data(), spoff.size() * sizeof(long long), cudaMemcpyHostToDevice));
      QBX_CUDA_TRY(cudaMemcpy(f->p2m_src.ptr, psrc.data(), psrc.size() * sizeof(int), cudaMemcpyHostToDevice));
      QBX_CUDA_TRY(cudaMemcpy(f->p2m_srcleaf.ptr, psleaf.data(), psleaf.size() * sizeof(int), cudaMemcpyHostToDevice));
    }
    QBX_CUDA_TRY(cudaMemcpy(f->p2m_lseg.ptr, lseg.data(), lseg.size() * sizeof(int), cudaMemcpyHostToDevice));
  }
  for (int b = 0; b < f->n_boxes; ++b)
    for (int e = xoff[b]; e < xoff[b + 1]; ++e) p2l += rs[xidx[e]].y - rs[xidx[e]].x;
  {  // P2L work items: each X box's sources, cut into pieces of one row chunk
    std::vector<int> xb(std::max(1, f->n_xbox));
    if (f->n_xbox)
      QBX_CUDA_TRY(cudaMemcpy(xb.data(), f->xbox.ptr, f->n_xbox * sizeof(int), cudaMemcpyDeviceToHost));
    const int pbx = max_order(f->h_pb, f->xbox_off);
    f->p2l_sm = rows_launch_smem(pbx);
    const int chunk = rows_chunk(pbx, f->p2l_sm);  // the least capacity over the X levels
    f->p2l_chunk = chunk;
    f->p2l_pb = pbx;
    std::vector<int> src, boff(f->n_xbox + 1, 0);
    std::vector<int4> items;
    std::vector<long long> poff;
    long long ptot = 0;
    for (int t = 0; t < f->n_xbox; ++t) {
      const int b = xb[t];
      const int Q = 2 * f->h_pb[blev[b]] + 1;
      const int s0 = (int)src.size();
      for (int e = xoff[b]; e < xoff[b + 1]; ++e)
        for (int i = rs[xidx[e]].x; i < rs[xidx[e]].y; ++i) src.push_back(i);
      boff[t] = (int)items.size();
      for (int a = s0; a < (int)src.size(); a += chunk) {
        items.push_back(make_int4(b, a, std::min(chunk, (int)src.size() - a), 0));
        poff.push_back(ptot);
        ptot += Q;
      }
    }
    boff[f->n_xbox] = (int)items.size();
    f->n_p2l_items = (int)items.size();
    QBX_CUDA_TRY(f->p2l_items.alloc(std::max<size_t>(1, items.size())));
    QBX_CUDA_TRY(f->p2l_poff.alloc(std::max<size_t>(1, poff.size())));
    QBX_CUDA_TRY(f->p2l_src.alloc(std::max<size_t>(1, src.size())));
    QBX_CUDA_TRY(f->p2l_boff.alloc(boff.size()));
    QBX_CUDA_TRY(f->p2l_part.alloc(std::max<long long>(1, ptot)));
    if (!items.empty()) {
      QBX_CUDA_TRY(cudaMemcpy(f->p2l_items.ptr, items.data(), items.size() * sizeof(int4), cudaMemcpyHostToDevice));
      QBX_CUDA_TRY(cudaMemcpy(f->p2l_poff.ptr, poff.data(), poff.size() * sizeof(long long), cudaMemcpyHostToDevice));
      QBX_CUDA_TRY(cudaMemcpy(f->p2l_src.ptr, src.data(), src.size() * sizeof(int), cudaMemcpyHostToDevice));
    }
    QBX_CUDA_TRY(cudaMemcpy(f->p2l_boff.ptr, boff.data(), boff.size() * sizeof(int), cudaMemcpyHostToDevice));
  }
  QBX_CUDA_TRY(f->src_leaves.alloc(std::max<size_t>(1, src_leaves.size())));
  if (!src_leaves.empty())
    QBX_CUDA_TRY(cudaMemcpy(f->src_leaves.ptr, src_leaves.data(), src_leaves.size() * 4,
                            cudaMemcpyHostToDevice));
  f->n_src_leaves = (int)src_leaves.size();
  h->stats[4] = f->n_boxes;
  h->stats[5] = f->n_leaves;
  h->stats[6] = f->n_levels - 1;
  h->stats[7] = f->pb_fine;
  h->stats[19] = f->pb_max;
  h->stats[8] = f->U.nnz;
  h->stats[9] = f->V.nnz;
  h->stats[10] = f->W.nnz;
  h->stats[11] = f->X.nnz;
  h->stats[12] = p2qbxl + w_direct_src;  // over all centres
  h->stats[13] = p2p;
  h->stats[14] = f->n_wpairs;
  h->stats[15] = m2p;
  h->stats[17] = p2l;
  {
    int64_t mm = 0;  // M2M and L2L translations (parents on levels >= 2)
    for (int b = 0; b < f->n_boxes; ++b)
      if (blev[b] >= 3) mm += 2;
    h->stats[18] = mm;
  }
  return QBX_OK;
}

namespace {

Fmm make_view(qbx_handle* h, FmmPlan* f, bool S, bool D) {
  Fmm F;
  F.level = f->box.level.ptr;
  F.child = f->box.child.ptr;
  F.centre = f->box.centre.ptr;
  F.rsrc = f->box.rng[PT_SRC].ptr;
  F.rctr = f->box.rng[PT_CTR].ptr;
  F.rtgt = f->box.rng[PT_TGT].ptr;
  F.uoff = f->U.off.ptr; F.uidx = f->U.idx.ptr;
  F.voff = f->V.off.ptr; F.vidx = f->V.idx.ptr; F.vcls = f->V_cls.ptr;
  F.woff = f->W.off.ptr; F.widx = f->W.idx.ptr;
  F.xoff = f->X.off.ptr; F.xidx = f->X.idx.ptr;
  F.sxy = f->s_xy.ptr; F.snrm = f->s_nrm.ptr; F.qs = f->qs.ptr; F.ds = f->ds.ptr;
  F.q32 = f->q32.ptr; F.ab32 = f->ab32.ptr; F.dn32 = f->dn32.ptr;
  F.qf = f->qf.ptr; F.df = f->df.ptr; F.nf = f->nf.ptr; F.sexp = f->sexp.ptr;
  F.cxy = f->c_xy.ptr; F.crad = f->c_r.ptr; F.cid = f->perm[PT_CTR].ptr;
  F.txy = f->t_xy.ptr; F.tid = f->perm[PT_TGT].ptr; F.tassoc = f->t_assoc.ptr;
  F.lpb = f->lpb.ptr; F.eoff = f->eoff.ptr;
  F.scale = f->scale.ptr; F.pw = f->pw.ptr; F.ipw = f->ipw.ptr;
  F.t_m2l = f->t_m2l.ptr; F.t_m2m = f->t_m2m.ptr; F.t_l2l = f->t_l2l.ptr;
  F.mpole = f->mpole.ptr; F.local = f->local.ptr; F.lpq = f->lpq.ptr;
  F.ffs = f->ff_s.ptr; F.loc32 = f->loc32.ptr;
  F.conv = f->conv.ptr; F.iconv = f->iconv.ptr; F.lsig = f->lsig.ptr; F.isig = f->isig.ptr; F.isf = f->isf.ptr; F.sigr = f->sigr.ptr;
  F.U = make_ff_units(h->k);
  F.k = h->k; F.ik = 1.0 / h->k; F.side = f->side; F.pbmax = f->pb_max; F.p = h->p; F.n_levels = f->n_levels;
  F.has_S = S ? 1 : 0; F.has_D = D ? 1 : 0;
  return F;
}

// L2QBXL at the centres of set C (adds to alpha).
qbx_status launch_l2qbxl(const Fmm& F, FmmPlan* f, qbx_handle* h, const CentreSet& C, cd* alpha,
                         bool mixed, cudaStream_t s) {
  if (C.n == 0) return QBX_OK;
  stage_begin(h, QBX_STAGE_L2QBXL, s);
  // a warp per G centres. G: up to 32 (every lane fills a row), but no more
  // than keeps about two warps per SM for a handle evaluated alone (the dot
  // products keep the FP64 pipe busy from one warp; batched handles share the
  // GPU), within the shared memory of the rows.
  {
    const int TW = f->cleaf_pb_max + h->p + 1;
    int G = 32;
    if (h->l2qbxl_g > 0) G = h->l2qbxl_g;  // set by an autotuner
    else
      while (!h->batched && G > 1 && (C.n + G - 1) / G < 152 * 2) G /= 2;
    // (batched handles share the SMs with other curves' stages and keep the
    // larger rows)
    const bool ff32 = mixed && f->ff_leaves;
    const size_t lim = (mixed && !h->batched) ? kL2qbxlMixedSmem : kL2qbxlSmem;
    const size_t slot = ff32 ? sizeof(float2) : sizeof(cd);
    while (G > 1 && (size_t)G * TW * slot > lim) G /= 2;
    const size_t sm = (size_t)G * TW * slot;
    if (ff32) {
      l2qbxl_ff_kernel<<<nblk(C.n, G), 32, sm, s>>>(F, f->cleaf.ptr, C.clist.ptr, C.n, G, TW, alpha);
    } else if (mixed) {
      split_coef_kernel<<<nblk(f->n_coef, 256), 256, 0, s>>>(f->local.ptr, f->n_coef, f->sp_m.ptr,
                                                             f->sp_e.ptr);
      l2qbxl_mixed_kernel<<<nblk(C.n, G), 32, sm, s>>>(F, f->cleaf.ptr, C.clist.ptr, C.n, G, TW,
                                                      f->sp_m.ptr, f->sp_e.ptr, alpha);
      h->launches += 1;
    } else {
      l2qbxl_kernel<<<nblk(C.n, G), 32, sm, s>>>(F, f->cleaf.ptr, C.clist.ptr, C.n, G, TW, alpha);
    }
  }
  QBX_KCHECK("l2qbxl", s);
  stage_end(h, QBX_STAGE_L2QBXL, s);
  h->launches += 1;
  return QBX_OK;
}

// M2QBXL at the centres of set C (adds to alpha).
template <int PM>
qbx_status launch_m2qbxl(const Fmm& F, FmmPlan* f, qbx_handle* h, bool S, bool D,
                         const CentreSet& C, cd* alpha, bool mixed, cudaStream_t s) {
  if (C.n == 0) return QBX_OK;
  stage_begin(h, QBX_STAGE_M2QBXL, s);
  if (C.n_pairs > 0 && (S || D)) {
    const int np = C.n_pairs;
    cd* part = f->wpart.ptr;
    // mixed: pairs per warp PW (at most kM2qbxlMixedPairs for a handle
    // evaluated alone, 32 for batched handles, which share the SMs with other
    // curves' stages) so that a warp's split rows (20 B per order) take at most
    // kM2qbxlMixedSmem, and, for a handle evaluated alone, fewer while that
    // leaves under two warps per SM (few pairs: spread the sequential
    // recurrences over all SMs)
    const int TW = C.wp_pbmax + h->p + 1;
    int PW = h->batched ? 32 : kM2qbxlMixedPairs;
    while (PW > 1 && (size_t)PW * TW * 20 > kM2qbxlMixedSmem) PW /= 2;
    while (!h->batched && PW > 1 && (np + PW - 1) / PW < 152 * 2) PW /= 2;
    if (mixed && f->ff_wboxes && (size_t)PW * TW * 16 <= kM2qbxlMixedSmem) {
      mpole_scaled_kernel<<<f->n_cw_box, kThreads, 0, s>>>(F, f->cw_box.ptr, f->sp_m.ptr);
      m2qbxl_ff_kernel<<<nblk(np, PW), 32, (size_t)PW * TW * 16, s>>>(
          F, C.wp_ctr.ptr, C.wp_box.ptr, np, PW, TW, f->sp_m.ptr, part);
      h->launches += 1;
    } else if (mixed && (size_t)PW * TW * 20 <= kM2qbxlMixedSmem) {
      const long long ncoef = f->n_coef;
      split_coef_kernel<<<nblk(ncoef, 256), 256, 0, s>>>(f->mpole.ptr, ncoef, f->sp_m.ptr,
                                                        f->sp_e.ptr);
      sf_split_kernel<<<f->n_levels, 64, 0, s>>>(F, f->sf_m.ptr, f->sf_e.ptr);
      m2qbxl_mixed_kernel<<<nblk(np, PW), 32, (size_t)PW * TW * 20, s>>>(
          F, C.wp_ctr.ptr, C.wp_box.ptr, np, PW, TW, f->sp_m.ptr, f->sp_e.ptr, f->sf_m.ptr,
          f->sf_e.ptr, part);
      h->launches += 2;
    } else {
      const int nparts = (2 * h->p + 1 + kM2qbxlOrders - 1) / kM2qbxlOrders;
      const unsigned gb = nblk((int64_t)np * nparts, kM2qbxlBlock);
      constexpr int B = kM2qbxlBlock;
      if (S && D) m2qbxl_pair_kernel<PM, true, true><<<gb, B, 0, s>>>(F, C.wp_ctr.ptr, C.wp_box.ptr, np, part);
      else if (S) m2qbxl_pair_kernel<PM, true, false><<<gb, B, 0, s>>>(F, C.wp_ctr.ptr, C.wp_box.ptr, np, part);
      else m2qbxl_pair_kernel<PM, false, true><<<gb, B, 0, s>>>(F, C.wp_ctr.ptr, C.wp_box.ptr, np, part);
    }
    QBX_KCHECK("m2qbxl", s);
    const int P = 2 * h->p + 1;
    m2qbxl_sum_kernel<<<nblk((int64_t)C.n * P, 256), 256, 0, s>>>(C.n, P, C.wp_off.ptr, part,
                                                                 f->perm[PT_CTR].ptr, C.clist.ptr,
                                                                 mixed ? f->sexp.ptr : nullptr,
                                                                 alpha);
    QBX_KCHECK("m2qbxl_sum", s);
    h->launches += 2;
  }
  stage_end(h, QBX_STAGE_M2QBXL, s);
  return QBX_OK;
}

// P2QBXL (U list and directly summed W boxes): one warp per centre, adds to alpha.
template <int PM>
qbx_status launch_centre_near(const Fmm& F, FmmPlan* f, qbx_handle* h, bool S, bool D,
                              const CentreSet& C, cd* alpha, bool mixed, cudaStream_t s) {
  if (!(S || D) || C.n == 0) return QBX_OK;
  stage_begin(h, QBX_STAGE_P2QBXL, s);
  const int nc = C.n;
  const int* cl = C.clist.ptr;
  auto launch = [&](auto w) {
    constexpr int W = decltype(w)::value;
    const int bt = nc < kSmallBlockCentres ? 32 : kThreads;
    const unsigned g = nblk(nc, bt / W);
#define P2QBXL_ARGS <<<g, bt, 0, s>>>(F, f->cleaf.ptr, f->wd_off.ptr, f->wd_box.ptr, cl, nc, alpha)
    if (mixed) {
      if (S && D) p2qbxl_warp_mixed_kernel<PM, true, true, W> P2QBXL_ARGS;
      else if (S) p2qbxl_warp_mixed_kernel<PM, true, false, W> P2QBXL_ARGS;
      else p2qbxl_warp_mixed_kernel<PM, false, true, W> P2QBXL_ARGS;
    } else {
      if (S && D) p2qbxl_warp_kernel<PM, true, true, W> P2QBXL_ARGS;
      else if (S) p2qbxl_warp_kernel<PM, true, false, W> P2QBXL_ARGS;
      else p2qbxl_warp_kernel<PM, false, true, W> P2QBXL_ARGS;
    }
#undef P2QBXL_ARGS
  };
  if (h->n_ctr >= kHalfWarpCentres) launch(std::integral_constant<int, 16>());
  else launch(std::integral_constant<int, 32>());
  QBX_KCHECK("p2qbxl", s);
  stage_end(h, QBX_STAGE_P2QBXL, s);
  h->launches += 1;
  return QBX_OK;
}


}  // namespace

namespace {

template <int PM>
qbx_status centre_near_dispatch(const Fmm& F, FmmPlan* f, qbx_handle* h, bool S, bool D,
                                const CentreSet& C, bool mixed, cudaStream_t s) {
  return launch_centre_near<PM>(F, f, h, S, D, C, h->alpha.ptr, mixed, s);
}

}  // namespace

// Stream organisation. Two streams: the caller's (main) and the plan's side
// stream. Every stage adds into zeroed outputs, and each output array is
// written by one stream at a time:
//   main: P2M, M2M | M2L (after P2L) | L2L, unscale | L2P (after M2P) |
//         L2QBXL (after the side stream)
//   side: zero alpha, out; P2L; P2QBXL; P2P | M2QBXL, M2P (after M2M)
// P2L needs only the strengths and adds into the locals before M2L does; the
// centre coefficients alpha are written by P2QBXL and M2QBXL (side) before
// L2QBXL (main); out is written by P2P and M2P (side) before L2P (main).
// L2QBXL follows L2P instead of running beside it: run concurrently, the two
// took longer than one after the other (2.62 against 2.10 ms for the whole
// step of the starfish k = 10 workload). With per-stage timing on, everything
// runs on the main stream in the same order, so that stage times do not
// overlap.
qbx_status fmm_eval(qbx_handle* h, bool S, bool D, cd* out, int precision, bool all_centres,
                    cudaStream_t s) {
  FmmPlan* f = h->fmm;
  if (!f) { set_error("FMM plan missing"); return QBX_ERR_STATE; }
  // alpha is formed at every centre when the caller asks for it, else only at
  // the centres some target is associated with (the only ones QBXL2P reads)
  const CentreSet& C = f->cset[all_centres ? 0 : 1];
  const std::vector<int>& pb = f->h_pb;
  const bool mixed = precision == QBX_MIXED;
  if (h->n_src > 0) {
    gather_strengths_kernel<<<nblk(h->n_src, 256), 256, 0, s>>>(
        h->n_src, f->perm[PT_SRC].ptr, h->q_str.ptr, h->d_str.ptr, f->s_nrm.ptr, h->k,
        f->qs.ptr, f->ds.ptr, mixed ? f->q32.ptr : nullptr, mixed ? f->ab32.ptr : nullptr,
        f->dn32.ptr, f->qf.ptr, f->df.ptr, f->nf.ptr, mixed ? h->str_exp.ptr : nullptr,
        (int)strength_blocks(h->n_src), f->sexp.ptr);
    QBX_KCHECK("gather_strengths", s);
    h->launches += 1;
  }
  Fmm F = make_view(h, f, S, D);
  QBX_CUDA_TRY(cudaMemsetAsync(f->mpole.ptr, 0, (size_t)f->n_coef * sizeof(cd), s));
  QBX_CUDA_TRY(cudaMemsetAsync(f->local.ptr, 0, (size_t)f->n_coef * sizeof(cd), s));
  const bool fork = !h->timing && !debug_sync() && !h->batched && f->near_stream != nullptr;
  cudaStream_t s2 = fork ? f->near_stream : s;
  auto signal = [&](cudaEvent_t ev, cudaStream_t from) -> qbx_status {
    if (fork) QBX_CUDA_TRY(cudaEventRecord(ev, from));
    return QBX_OK;
  };
  auto wait = [&](cudaStream_t on, cudaEvent_t ev) -> qbx_status {
    if (fork) QBX_CUDA_TRY(cudaStreamWaitEvent(on, ev, 0));
    return QBX_OK;
  };
  TRY(signal(f->ev_fork, s));
  TRY(wait(s2, f->ev_fork));
  const int P = 2 * h->p + 1;
  // ---- side: zero the outputs, P2L, then the near field
  if (h->n_ctr > 0) QBX_CUDA_TRY(cudaMemsetAsync(h->alpha.ptr, 0, (size_t)h->n_ctr * P * sizeof(cd), s2));
  if (h->n_tgt > 0) QBX_CUDA_TRY(cudaMemsetAsync(out, 0, (size_t)h->n_tgt * sizeof(cd), s2));
  stage_begin(h, QBX_STAGE_P2L, s2);
  if ((S || D) && f->n_p2l_items > 0) {  // X lists without sources add nothing
    if (mixed)
      p2l_item_mixed_kernel<<<f->n_p2l_items, kP2lMixedThreads,
                              p2l_mixed_smem(f->p2l_pb, f->p2l_chunk), s2>>>(
          F, f->p2l_items.ptr, f->p2l_src.ptr, f->p2l_poff.ptr, f->p2l_part.ptr, f->p2l_chunk,
          f->m2p_rec.ptr);
    else
      p2l_item_kernel<<<f->n_p2l_items, kThreads, f->p2l_sm, s2>>>(
          F, f->p2l_items.ptr, f->p2l_src.ptr, f->p2l_poff.ptr, f->p2l_part.ptr, (unsigned)f->p2l_sm);
    QBX_KCHECK("p2l", s2);
    p2l_sum_kernel<<<f->n_xbox, kThreads, 0, s2>>>(F, f->xbox.ptr, f->p2l_boff.ptr, f->p2l_poff.ptr,
                                                  f->p2l_part.ptr);
    QBX_KCHECK("p2l_sum", s2);
    h->launches += 2;
  }
  stage_end(h, QBX_STAGE_P2L, s2);
  TRY(signal(f->ev_p2l, s2));
  if (h->n_ctr > 0) {
    if (h->p <= 4) TRY(centre_near_dispatch<4>(F, f, h, S, D, C, mixed, s2));
    else if (h->p <= 8) TRY(centre_near_dispatch<8>(F, f, h, S, D, C, mixed, s2));
    else if (h->p <= 12) TRY(centre_near_dispatch<12>(F, f, h, S, D, C, mixed, s2));
    else TRY(centre_near_dispatch<16>(F, f, h, S, D, C, mixed, s2));
  }
  stage_begin(h, QBX_STAGE_P2P, s2);
  if (f->n_utgt > 0 && (S || D)) {
    const unsigned gw = nblk(f->n_utgt, kThreads / 32);  // one warp per target
#define P2P_LAUNCH(A, B)                                                                      \
    do {                                                                                       \
      if (mixed)                                                                               \
        p2p_warp_mixed_kernel<A, B><<<gw, kThreads, 0, s2>>>(F, f->utgt.ptr, f->tleaf.ptr,     \
                                                             f->n_utgt, out);                  \
      else                                                                                     \
        p2p_warp_kernel<A, B><<<gw, kThreads, 0, s2>>>(F, f->utgt.ptr, f->tleaf.ptr,           \
                                                       f->n_utgt, out);                        \
    } while (0)
    if (S && D) P2P_LAUNCH(true, true);
    else if (S) P2P_LAUNCH(true, false);
    else P2P_LAUNCH(false, true);
#undef P2P_LAUNCH
    QBX_KCHECK("p2p", s2);
    h->launches += 1;
  }
  stage_end(h, QBX_STAGE_P2P, s2);
  // ---- main: upward pass
  stage_begin(h, QBX_STAGE_P2M, s);
  if ((S || D) && f->n_p2m_items > 0) {
    if (mixed) {
      p2m_item_mixed_kernel<<<f->n_p2m_items, kP2mMixedThreads,
                              p2m_mixed_smem(f->p2m_pb, f->p2m_chunk), s>>>(
          F, f->p2m_items.ptr, f->p2m_segleaf.ptr, f->p2m_segrow.ptr, f->p2m_segpoff.ptr,
          f->p2m_src.ptr, f->p2m_srcleaf.ptr, f->p2m_part.ptr, f->p2m_chunk);
      QBX_KCHECK("p2m", s);
      p2m_sum_mixed_kernel<<<f->n_src_leaves, kThreads, 0, s>>>(
          F, f->src_leaves.ptr, f->p2m_lseg.ptr, f->p2m_segpoff.ptr, f->p2m_part.ptr);
    } else {
      p2m_item_kernel<<<f->n_p2m_items, kThreads, f->p2m_sm, s>>>(
          F, f->p2m_items.ptr, f->p2m_segleaf.ptr, f->p2m_segrow.ptr, f->p2m_segpoff.ptr,
          f->p2m_src.ptr, f->p2m_srcleaf.ptr, f->p2m_part.ptr, (unsigned)f->p2m_sm);
      QBX_KCHECK("p2m", s);
      p2m_sum_kernel<<<f->n_src_leaves, kThreads, 0, s>>>(F, f->src_leaves.ptr, f->p2m_lseg.ptr,
                                                         f->p2m_segpoff.ptr, f->p2m_part.ptr);
    }
    QBX_KCHECK("p2m_sum", s);
    h->launches += 2;
  }
  stage_end(h, QBX_STAGE_P2M, s);
  stage_begin(h, QBX_STAGE_M2M, s);
  if (mixed) {
    TRY(launch_m2m_f32(h, f, s));
  } else {
    for (int l = f->n_levels - 2; l >= 2; --l) {
      const int nb = f->nonleaf_off[l + 1] - f->nonleaf_off[l];
      if (nb == 0) continue;
      m2m_kernel<<<dim3(nb, fold_split(nb, 2 * pb[l] + 1)), kThreads, m2m_smem(pb[l + 1]), s>>>(
          F, f->nonleaf.ptr + f->nonleaf_off[l], f->tmm_f64.ptr + f->h_fold_off[l]);
      QBX_KCHECK("m2m", s);
      h->launches += 1;
    }
  }
  stage_end(h, QBX_STAGE_M2M, s);
  TRY(signal(f->ev_m2m, s));
  // ---- side: W-list stages (need the multipoles)
  TRY(wait(s2, f->ev_m2m));
  if (h->n_ctr > 0) {
    cd* alpha = h->alpha.ptr;
    if (h->p <= 4) TRY(launch_m2qbxl<4>(F, f, h, S, D, C, alpha, mixed, s2));
    else if (h->p <= 8) TRY(launch_m2qbxl<8>(F, f, h, S, D, C, alpha, mixed, s2));
    else if (h->p <= 12) TRY(launch_m2qbxl<12>(F, f, h, S, D, C, alpha, mixed, s2));
    else TRY(launch_m2qbxl<16>(F, f, h, S, D, C, alpha, mixed, s2));
  }
  stage_begin(h, QBX_STAGE_M2P, s2);
  if (f->n_wtgt > 0 && f->n_m2p_pairs > 0) {
    if (mixed) {
      mpole_f32_list_kernel<<<f->n_m2p_wbox, kThreads, 0, s2>>>(
          F, f->m2p_wbox.ptr, f->conv.ptr, f->m2p_mu.ptr);
      QBX_KCHECK("m2p_mu", s2);
      m2p_pair_mixed_kernel<<<nblk(f->n_m2p_pairs, kThreads), kThreads, 0, s2>>>(
          F, f->m2p_tgt.ptr, f->m2p_box.ptr, f->m2p_slot.ptr, f->n_m2p_pairs, f->m2p_mu.ptr,
          f->m2p_rec.ptr, reinterpret_cast<float4*>(f->m2p_part.ptr));
      QBX_KCHECK("m2p", s2);
      m2p_sum_mixed_kernel<<<nblk(f->n_wtgt, kThreads), kThreads, 0, s2>>>(
          f->n_wtgt, f->wtgt.ptr, f->m2p_off.ptr, reinterpret_cast<float4*>(f->m2p_part.ptr),
          f->perm[PT_TGT].ptr, f->sexp.ptr, out);
    } else {
      mpole_pq_kernel<<<f->n_m2p_wbox, kThreads, 0, s2>>>(F, f->m2p_wbox.ptr, f->m2p_big.ptr,
                                                         f->m2p_pq.ptr);
      QBX_KCHECK("m2p_pq", s2);
      m2p_pair_kernel<<<nblk(f->n_m2p_pairs, kThreads), kThreads, 0, s2>>>(
          F, f->m2p_tgt.ptr, f->m2p_box.ptr, f->m2p_slot.ptr, f->n_m2p_pairs, f->m2p_big.ptr,
          f->m2p_pq.ptr, f->m2p_part.ptr);
      QBX_KCHECK("m2p", s2);
      m2p_sum_kernel<<<nblk(f->n_wtgt, kThreads), kThreads, 0, s2>>>(
          f->n_wtgt, f->wtgt.ptr, f->m2p_off.ptr, f->m2p_part.ptr, f->perm[PT_TGT].ptr, out);
    }
    QBX_KCHECK("m2p_sum", s2);
    h->launches += 3;
  }
  stage_end(h, QBX_STAGE_M2P, s2);
  TRY(signal(f->ev_out, s2));
  // ---- main: downward pass (M2L after P2L has added into the locals)
  TRY(wait(s, f->ev_p2l));
  stage_begin(h, QBX_STAGE_M2L, s);
  // tensor cores for the FP64 path; the mixed path keeps the FP32 CUDA-core
  // tile GEMM (faster on every measured workload) unless engine 1 asks for them
  if (f->tc_any && (!mixed || h->m2l_engine == 1)) {
    TRY(launch_m2l_tc(h, f, mixed, s));
  } else if (mixed) {
    TRY(launch_m2l_f32(h, f, s));
  } else {
    TRY(launch_m2l_f64(h, f, s));
  }
  stage_end(h, QBX_STAGE_M2L, s);
  stage_begin(h, QBX_STAGE_L2L, s);
  if (mixed) {
    TRY(launch_l2l_f32(h, f, s));
  } else {
    for (int l = 2; l + 1 < f->n_levels; ++l) {
      const int nb = f->nonleaf_off[l + 1] - f->nonleaf_off[l];
      if (nb == 0) continue;
      l2l_kernel<<<dim3(nb, fold_split(nb, 2 * pb[l + 1] + 1)), kThreads, l2l_smem(pb[l]), s>>>(
          F, f->nonleaf.ptr + f->nonleaf_off[l], f->tl_f64.ptr + f->h_fold_off[l]);
      QBX_KCHECK("l2l", s);
      h->launches += 1;
    }
  }
  if (f->n_leaves > 0) {
    unscale_leaf_locals_kernel<<<nblk(f->n_leaves, kBoxGroup), kThreads, 0, s>>>(
        F, f->leaves.ptr, f->n_leaves, mixed);
    QBX_KCHECK("unscale_leaf_locals", s);
    h->launches += 1;
  }
  stage_end(h, QBX_STAGE_L2L, s);
  // ---- main: L2P (out, after M2P), then L2QBXL (alpha, after the side stream)
  TRY(signal(f->ev_join, s2));
  TRY(wait(s, f->ev_out));
  if (f->n_dtgt > 0) {
    stage_begin(h, QBX_STAGE_L2P, s);
    if (mixed)
      l2p_mixed_kernel<<<nblk(f->n_dtgt, kThreads), kThreads, 0, s>>>(F, f->dtgt.ptr, f->tleaf.ptr,
                                                                      f->n_dtgt, out);
    else
      l2p_kernel<<<nblk(f->n_dtgt, kThreads), kThreads, 0, s>>>(F, f->dtgt.ptr, f->tleaf.ptr,
                                                                f->n_dtgt, out);
    QBX_KCHECK("l2p", s);
    stage_end(h, QBX_STAGE_L2P, s);
    h->launches += 1;
  }
  TRY(wait(s, f->ev_join));
  if (h->n_ctr > 0) {
    cd* alpha = h->alpha.ptr;
    TRY(launch_l2qbxl(F, f, h, C, alpha, mixed, s));
  }
  QBX_CUDA_TRY(cudaGetLastError());
  return QBX_OK;
}

void fmm_plan_free(FmmPlan* f) {
  DeviceQuiet quiet;
  delete f;
}

extern "C" qbx_status qbx_export_tree(const qbx_handle* h, int64_t* info, double* root,
                                      int32_t* box_level, int32_t* box_ij, int32_t* box_child,
                                      int32_t* box_range, int32_t* lists_off,
                                      int32_t* lists_idx, int32_t* perm_src, int32_t* perm_ctr,
                                      int32_t* perm_tgt) {
  if (!h) { set_error("qbx_export_tree: NULL handle"); return QBX_ERR_ARG; }
  const FmmPlan* f = h->fmm;
  if (!f || !h->planned || h->mode != QBX_FMM) {
    set_error("qbx_export_tree: no FMM plan (call qbx_tree_build with QBX_FMM)");
    return QBX_ERR_STATE;
  }
  const int nb = f->n_boxes;
  if (info) {
    info[0] = nb; info[1] = f->n_levels; info[2] = f->U.nnz; info[3] = f->V.nnz;
    info[4] = f->W.nnz; info[5] = f->X.nnz; info[6] = f->pb_fine; info[7] = f->n_leaves;
  }
  if (root) { root[0] = f->x0; root[1] = f->y0; root[2] = f->side; }
  if (box_level) QBX_CUDA_TRY(cudaMemcpy(box_level, f->box.level.ptr, nb * 4, cudaMemcpyDeviceToHost));
  if (box_ij) QBX_CUDA_TRY(cudaMemcpy(box_ij, f->box.ij.ptr, nb * 8, cudaMemcpyDeviceToHost));
  if (box_child) QBX_CUDA_TRY(cudaMemcpy(box_child, f->box.child.ptr, (size_t)nb * 16, cudaMemcpyDeviceToHost));
  if (box_range) {
    std::vector<int2> r(nb);
    for (int t = 0; t < PT_COUNT; ++t) {
      QBX_CUDA_TRY(cudaMemcpy(r.data(), f->box.rng[t].ptr, (size_t)nb * 8, cudaMemcpyDeviceToHost));
      for (int b = 0; b < nb; ++b) {
        box_range[(size_t)b * 8 + 2 * t] = r[b].x;
        box_range[(size_t)b * 8 + 2 * t + 1] = r[b].y;
      }
    }
  }
  const Csr* L[4] = {&f->U, &f->V, &f->W, &f->X};
  size_t pos = 0;
  for (int i = 0; i < 4; ++i) {
    if (lists_off)
      QBX_CUDA_TRY(cudaMemcpy(lists_off + (size_t)i * (nb + 1), L[i]->off.ptr, (nb + 1) * 4,
                              cudaMemcpyDeviceToHost));
    if (lists_idx && L[i]->nnz)
      QBX_CUDA_TRY(cudaMemcpy(lists_idx + pos, L[i]->idx.ptr, L[i]->nnz * 4, cudaMemcpyDeviceToHost));
    pos += L[i]->nnz;
  }
  if (perm_src && h->n_src) QBX_CUDA_TRY(cudaMemcpy(perm_src, f->perm[PT_SRC].ptr, h->n_src * 4, cudaMemcpyDeviceToHost));
  if (perm_ctr && h->n_ctr) QBX_CUDA_TRY(cudaMemcpy(perm_ctr, f->perm[PT_CTR].ptr, h->n_ctr * 4, cudaMemcpyDeviceToHost));
  if (perm_tgt && h->n_tgt) QBX_CUDA_TRY(cudaMemcpy(perm_tgt, f->perm[PT_TGT].ptr, h->n_tgt * 4, cudaMemcpyDeviceToHost));
  return QBX_OK;
}

extern "C" qbx_status qbx_get_box_orders(const qbx_handle* h, int32_t* pb_out, int32_t n) {
  if (!h || !pb_out || n < 0) { set_error("qbx_get_box_orders: bad arguments"); return QBX_ERR_ARG; }
  const FmmPlan* f = h->fmm;
  if (!f || !h->planned || h->mode != QBX_FMM) {
    set_error("qbx_get_box_orders: no FMM plan (call qbx_tree_build with QBX_FMM)");
    return QBX_ERR_STATE;
  }
  for (int l = 0; l < n; ++l) pb_out[l] = l < f->n_levels ? f->h_pb[l] : 0;
  return QBX_OK;
}
