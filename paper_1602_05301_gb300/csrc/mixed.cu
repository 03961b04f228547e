// Mixed-precision kernels (QBX_MIXED): the M2M translation of Stage 2, the M2L
// translation of Stage 4 and the L2L translation of Stage 7 in complex FP32
// with compensated (Kahan) accumulation.
//
// FP32 cannot hold the power-scaled expansions of the FP64 path (their
// translation entries still grow like a factorial), so the FP32 operators act
// on sigma-normalised coefficients
//     mu_n = a_n / sig_|n|,   lam_l = gamma_l sig_|l|,
//     sig_j = min(1, (x/2)^j / j!),  x = k * side  (the size of J_j at a box),
// for which every M2L entry sig_l sig_n (-1)^l W_{n+l}(D) is of order one or
// smaller, and so is every L2L entry (sig'_s / sig_n) (-1)^{s-n} V_{s-n}(d)
// (sig' of the child level) and M2M entry (sig_n / sig'_s) conj(V_{s-n}(d))
// (sig' of the parent level): the scale ratios are binomial-sized while
// J_{s-n}(k d) decays factorially. The entries are computed in FP64 (through logarithms
// of the scale factors), with the angles of the offsets taken out, and stored as FP32
// matrices, two per (level, distance) for M2L and one per level for M2M and for L2L; the
// coefficient conversions between the two normalisations are FP64.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "f32x2.cuh"
#include "ff.cuh"
#include "tree.cuh"
#include "m2l_entry.cuh"

namespace {

constexpr int kT = 128;

inline unsigned nblk(int64_t n, int b) { return (unsigned)std::max<int64_t>(1, (n + b - 1) / b); }

// per level: lsig[j] = log sig_j, conv[j] = s^j / sig_j  (j = 0..pb_l; stride
// pbmax + 1), iconv = 1 / conv, isig[j] = 1 / sig_min(j, pb_l) (j = 0..pb_l + 1; stride
// pbmax + 2). isig is held at e^kMaxLogIsig = 1e299: orders it would exceed that at lie
// above 45 (the plan bounds s^pb), where a box's own points (0.71 sides away) and its
// nearest partners (1.5 sides) leave less than (0.71 / 1.5)^45 = 2e-15 of a potential.
constexpr double kMaxLogIsig = 690.0;
__global__ void sigma_tables_kernel(int n_levels, int pbmax, const int* __restrict__ lpb,
                                    double k, double side, const double* __restrict__ scale,
                                    double* __restrict__ lsig, double* __restrict__ conv,
                                    double* __restrict__ iconv, double* __restrict__ isig) {
  const int l = blockIdx.x, pb = lpb[l];
  const double x = k * side / (double)(1 << l);
  const double ls = log(scale[l]);
  for (int j = threadIdx.x; j <= pb; j += blockDim.x) {
    const double v = fmin(0.0, j * log(0.5 * x) - lgamma((double)j + 1.0));
    lsig[(size_t)l * (pbmax + 1) + j] = v;
    const double c = exp(j * ls - v);
    conv[(size_t)l * (pbmax + 1) + j] = c;
    iconv[(size_t)l * (pbmax + 1) + j] = 1.0 / c;
    const double i = exp(fmin(-v, kMaxLogIsig));
    isig[(size_t)l * (pbmax + 2) + j] = i;
    if (j == pb) isig[(size_t)l * (pbmax + 2) + pb + 1] = i;
  }
}

// Recurrence factors of G_m = sig_m H_m on level l (mixed M2P and P2L):
// rec[m] = (2m sig_{m+1} / sig_m, sig_{m+1} / sig_{m-1}) for 1 <= m < pb_l,
// rec[0] = (sig_1, 0), and rec[pb_l] with sig_{pb+1} taken as sig_pb.
__global__ void m2p_rec_kernel(int n_levels, int pbmax, const int* __restrict__ lpb,
                               const double* __restrict__ lsig, double2* __restrict__ rec) {
  const int l = blockIdx.x;
  if (l >= n_levels) return;
  const double* sg = lsig + (size_t)l * (pbmax + 1);
  double2* r = rec + (size_t)l * (pbmax + 2);
  const int pb = lpb[l];
  for (int m = threadIdx.x; m <= pbmax + 1; m += blockDim.x) {
    double2 v = make_double2(0.0, 0.0);
    if (m == 0 && pb >= 1) v.x = exp(sg[1]);
    if (m >= 1 && m < pb)
      v = make_double2(2.0 * m * exp(sg[m + 1] - sg[m]), exp(sg[m + 1] - sg[m - 1]));
    // one order beyond pb, normalised by sig_pb (mixed P2L's dipole terms)
    if (m == pb && pb >= 1) v = make_double2(2.0 * m, exp(sg[m] - sg[m - 1]));
    r[m] = v;
  }
}

// r[l][m] = (sig_{m-1} / sig_m, sig_{m+1} / sig_m) of level l, 1 where the
// neighbour order is outside 0..pb (the mixed P2M's dipole terms)
__global__ void sig_ratio_kernel(int n_levels, int pbmax, const int* __restrict__ lpb,
                                 const double* __restrict__ lsig, double2* __restrict__ r) {
  const int l = blockIdx.x;
  if (l >= n_levels) return;
  const double* sg = lsig + (size_t)l * (pbmax + 1);
  const int pb = lpb[l];
  for (int m = threadIdx.x; m <= pbmax + 1; m += blockDim.x) {
    double2 v = make_double2(1.0, 1.0);
    if (m <= pb) {
      if (m >= 1) v.x = exp(sg[m - 1] - sg[m]);
      else v.x = exp(sg[1 <= pb ? 1 : 0] - sg[0]);  // |0 - 1| = 1
      if (m + 1 <= pb) v.y = exp(sg[m + 1] - sg[m]);
    }
    r[(size_t)l * (pbmax + 2) + m] = v;
  }
}

// The FP32 M2L matrices. An offset D = |D| e^{i phi} acts on sigma-normalised
// coefficients as T[n][l] = (-1)^l sig_l sig_n W_{n+l}(D), W_m = H_m(k |D|) e^{i m phi}.
// With x_n = e^{i n phi} mu_n the angle is gone, and because H_{-m} = (-1)^m H_m the
// matrix splits into one for the even parts e_n = x_n + (-1)^n x_{-n} and one for the
// odd parts o_n = x_n - (-1)^n x_{-n} (0 <= n, l <= pb; e_0 = x_0):
//   y_l    = (-1)^l e^{ i l phi} (E_l + O_l),   E_l = sum_n Te[n][l] e_n,
//   y_{-l} =        e^{-i l phi} (E_l - O_l),   O_l = sum_n To[n][l] o_n,
//   Te, To = sig_l sig_n (H_{n+l} +- (-1)^l H_{n-l}) / 2:
// half the products, and the 40 offsets of a V list share the matrices of their
// kM2lDist distances. Tm[d][2][n][l] of level l here; grid (d, n), threads over l.
constexpr int kM2lDist = 7;  // |D| of (2,0) (2,1) (2,2) (3,0) (3,1) (3,2) (3,3) box sides
__host__ __device__ constexpr int m2l_dist(int cls) {  // of offset class (dx + 3) * 7 + dy + 3
  const int dx = cls / 7 - 3, dy = cls % 7 - 3;
  const int ax = dx < 0 ? -dx : dx, ay = dy < 0 ? -dy : dy;
  const int hi = ax > ay ? ax : ay, lo = ax > ay ? ay : ax;
  return hi == 2 ? lo : hi == 3 ? 3 + lo : -1;
}
__global__ void m2l_fold_matrix_kernel(int l, int pb, int pbmax, const cd* __restrict__ t_m2l,
                                       const double* __restrict__ scale,
                                       const double* __restrict__ lsig, float2* __restrict__ Tm) {
  const int d = blockIdx.x, n = blockIdx.y, P = pb + 1;
  const int dx = d < 3 ? 2 : 3, dy = d < 3 ? d : d - 3;
  const M2lNorm nm(t_m2l, scale, lsig, l, (dx + 3) * 7 + dy + 3, pbmax);
  const double turn = -atan2((double)dy, (double)dx) * 0.31830988618379067154;  // -phi / pi
  float2* te = Tm + ((size_t)2 * d * P + n) * P;
  float2* to = te + (size_t)P * P;
  for (int lo = threadIdx.x; lo <= pb; lo += blockDim.x) {
    cd ra, rb;
    sincospi((n + lo) * turn, &ra.y, &ra.x);
    sincospi((n - lo) * turn, &rb.y, &rb.x);
    cd a = cmul(nm.entry(n, lo), ra);         // (-1)^lo sig sig H_{n+lo}
    const cd b = cmul(nm.entry(n, -lo), rb);  // (-1)^lo sig sig H_{n-lo}
    if (lo & 1) a = mk(-a.x, -a.y);
    te[lo] = make_float2((float)(0.5 * (a.x + b.x)), (float)(0.5 * (a.y + b.y)));
    to[lo] = make_float2((float)(0.5 * (a.x - b.x)), (float)(0.5 * (a.y - b.y)));
  }
}
// rot[cls][m] = e^{i m phi}, m <= pbmax
__global__ void m2l_rot_kernel(int pbmax, float2* __restrict__ rot) {
  const int cls = blockIdx.x;
  const double turn = atan2((double)(cls % 7 - 3), (double)(cls / 7 - 3)) * 0.31830988618379067154;
  for (int m = threadIdx.x; m <= pbmax; m += blockDim.x) {
    double c, sn;
    sincospi(m * turn, &sn, &c);
    rot[(size_t)cls * (pbmax + 1) + m] = make_float2((float)c, (float)sn);
  }
}

// isf[l][j] = 2^{s j} / sig_min(j, pb) as a pair of FP32, s = ffs[l] (0 on levels
// without), from the logarithm: it fits FP32 (float_float_scale) where 1 / sig_j is
// beyond FP64
__global__ void isig_ff_kernel(int n_levels, int pbmax, const int* __restrict__ lpb,
                               const int* __restrict__ ffs, const double* __restrict__ lsig,
                               float2* __restrict__ isf) {
  const int l = blockIdx.x;
  if (l >= n_levels) return;
  const int s = ffs[l];
  for (int j = threadIdx.x; j < pbmax + 2; j += blockDim.x) {
    float2 v = make_float2(0.f, 0.f);
    if (s != kNoFf && j <= lpb[l] + 1) {
      const double x = exp(fma((double)(s * j), 0.69314718055994530942,
                               -lsig[(size_t)l * (pbmax + 1) + min(j, lpb[l])]));
      v.x = (float)x;
      v.y = (float)(x - (double)v.x);
    }
    isf[(size_t)l * (pbmax + 2) + j] = v;
  }
}

__device__ __forceinline__ void kahan_add(float& s, float& c, float v) {
  const float y = v - c;
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}

// The tile GEMMs. A CTA takes some rows (M2L: V-list pairs; M2M, L2L: parents) that
// share a matrix: their FP32 coefficients go to shared memory ([n][row], n-major), and
// each thread computes one output order for R rows, streaming the matrix once for all
// of them. Sums: plain FP32 FMAs over blocks of kGemmBlock terms, blocks added with
// Kahan compensation.
constexpr int kGemmRows = 16;
constexpr int kGemmBlock = 8;
// Complex products of M2L between Kahan steps: with eight the rotated form's error
// against FP64 was 1.71e-7, with four 1.62e-7 (1.75e-7 with one matrix per offset class;
// now, with M2M and L2L rounded once per level, 1.51e-7), at 2.32 ms instead of 2.21 on
// 200 ellipses. (Relative l2, geometric mean over the four mixed cases that
// perf/cases.py lists and the first fourteen FMM evaluations that it draws from
// random.Random(77), in mixed precision, inputs of seed 5.)
constexpr int kKahanBlock = 4;
// Staged rows: order n of the row pair (r, r + 1), r even, is the float4 (re r,
// re r+1, im r, im r+1) at x + n * stage_stride(R) + r, so that each half is an
// operand of the packed FMAs. Two float2 of padding per n keep the row pairs
// 16-byte aligned and spread the staging stores over the banks.
__host__ __device__ constexpr int stage_stride(int R) { return R + 2; }
__device__ __forceinline__ void stage_put(float2* x, size_t n, int r, int RS, float2 v) {
  float* f = reinterpret_cast<float*>(x + n * RS + (r & ~1)) + (r & 1);
  f[0] = v.x;
  f[2] = v.y;
}

// Sums of R rows, row pairs packed: value s, lost part n (the sum is s + n).
template <int R>
struct RowSums {
  f32p sr[R / 2], si[R / 2], nr[R / 2], ni[R / 2];
  __device__ __forceinline__ RowSums() {
#pragma unroll
    for (int r = 0; r < R / 2; ++r) sr[r] = si[r] = nr[r] = ni[r] = 0ull;
  }
  __device__ __forceinline__ float sum_r(int r) const { return part(sr[r / 2], r); }
  __device__ __forceinline__ float sum_i(int r) const { return part(si[r / 2], r); }
  __device__ __forceinline__ float lost_r(int r) const { return part(nr[r / 2], r); }
  __device__ __forceinline__ float lost_i(int r) const { return part(ni[r / 2], r); }
  __device__ static __forceinline__ float part(f32p v, int r) {
    const float2 u = unpk(v);
    return (r & 1) ? u.y : u.x;
  }
};

// nj (1 <= nj <= kGemmBlock) terms of a tile product column, S += sum_{j < nj}
// tb[j] * x[j]: every kKahanBlock of them summed from the lost part of S and added to S
// (Kahan compensation in three operations).
template <int R>
__device__ __forceinline__ void gemm_block_add(const float2 (&tb)[kGemmBlock], int nj,
                                               const float2* __restrict__ x, RowSums<R>& S) {
  static_assert(R % 2 == 0, "rows are read in pairs");
  constexpr int RS = stage_stride(R);
  f32p tr[R / 2], ti[R / 2];
#pragma unroll
  for (int j = 0; j < kGemmBlock; ++j) {
    if (j < nj) {
      const f32p tx = pk(tb[j].x, tb[j].x), ty = pk(tb[j].y, tb[j].y);
      const f32p my = pk(-tb[j].y, -tb[j].y);
      const ulonglong2* m = reinterpret_cast<const ulonglong2*>(x + j * RS);
#pragma unroll
      for (int r = 0; r < R / 2; ++r) {
        const ulonglong2 v = m[r];  // (re, re), (im, im) of rows 2r, 2r + 1
        if (j > 0 && j % kKahanBlock == 0) {
          kahan_add2(S.sr[r], S.nr[r], tr[r]);
          kahan_add2(S.si[r], S.ni[r], ti[r]);
        }
        if (j % kKahanBlock == 0) {
          tr[r] = fma2(tx, v.x, fma2(my, v.y, S.nr[r]));
          ti[r] = fma2(tx, v.y, fma2(ty, v.x, S.ni[r]));
        } else {
          tr[r] = fma2(tx, v.x, fma2(my, v.y, tr[r]));
          ti[r] = fma2(tx, v.y, fma2(ty, v.x, ti[r]));
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < R / 2; ++r) {
    kahan_add2(S.sr[r], S.nr[r], tr[r]);
    kahan_add2(S.si[r], S.ni[r], ti[r]);
  }
}

// One output column lo of a tile product: for every row r < R,
// S[r] += sum_{n < N} M[n * ld + lo] * x[n][r], with x in shared memory (16-byte
// aligned, stage_put's layout). Packed FP32 FMAs over blocks of kGemmBlock terms
// (whose matrix entries are loaded one block ahead, into two alternating
// register sets), the blocks added with Kahan compensation. Threads with
// act == false read column 0 and their sums are not used.
template <int R = kGemmRows>
__device__ __forceinline__ void tile_gemm_column(const float2* __restrict__ M, size_t ld, int N,
                                                 const float2* __restrict__ x, int lo, bool act,
                                                 RowSums<R>& S) {
  constexpr int RS = stage_stride(R);
  const float2* Mc = M + (act ? lo : 0);
  const int nfull = N - N % kGemmBlock;
  float2 ba[kGemmBlock], bb[kGemmBlock];
  if (nfull > 0) {
#pragma unroll
    for (int j = 0; j < kGemmBlock; ++j) ba[j] = Mc[(size_t)j * ld];
  }
  for (int n0 = 0; n0 < nfull; n0 += 2 * kGemmBlock) {
    const int n1 = n0 + kGemmBlock;
    if (n1 < nfull) {
#pragma unroll
      for (int j = 0; j < kGemmBlock; ++j) bb[j] = Mc[(size_t)(n1 + j) * ld];
    }
    gemm_block_add<R>(ba, kGemmBlock, x + n0 * RS, S);
    if (n1 >= nfull) break;
    if (n1 + kGemmBlock < nfull) {
#pragma unroll
      for (int j = 0; j < kGemmBlock; ++j) ba[j] = Mc[(size_t)(n1 + kGemmBlock + j) * ld];
    }
    gemm_block_add<R>(bb, kGemmBlock, x + n1 * RS, S);
  }
  if (nfull < N) {  // the last, partial block
    const int nj = N - nfull;
#pragma unroll
    for (int j = 0; j < kGemmBlock; ++j)
      ba[j] = j < nj ? Mc[(size_t)(nfull + j) * ld] : make_float2(0.f, 0.f);
    gemm_block_add<R>(ba, nj, x + nfull * RS, S);
  }
}

// Programmatic dependent launch: a kernel launched with the attribute starts while
// its predecessor in the stream still runs, prepares what does not depend on it
// and waits here for its completion; the predecessor allows that at its start.
// Both are no-ops in an ordinary launch.
__device__ __forceinline__ void pdl_allow_next() {
  asm volatile("griddepcontrol.launch_dependents;");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The sigma-normalised multipoles mu_n = mh_n conv_|n| of the boxes that are V-list
// sources, as the FP32 sums that m2l_fold_kernel turns by a pair's angle: float4
// (mu_n + (-1)^n mu_{-n}, mu_n - (-1)^n mu_{-n}), n = 0..pb (mu_0, 0 at n = 0), at
// entry eoff[b] + b of mu32.
// kBoxGroup boxes per CTA, their orders side by side over its threads: one box's pb + 1
// orders would leave a last warp nearly empty, and the FP64 pipe takes as long for it
// (M2L with this of 200 ellipses 2.41 -> 2.36 ms).
__global__ void __launch_bounds__(kT) mpole_to_f32_kernel(
    int pbmax, const int* __restrict__ boxes, int n_boxes, const int* __restrict__ level,
    const int* __restrict__ lpb, const long long* __restrict__ eoff,
    const double* __restrict__ conv, const cd* __restrict__ mpole, float2* __restrict__ mu32) {
  __shared__ BoxGroup g;
  g.fill(boxes, n_boxes, level, lpb);
  for (int idx = threadIdx.x, u = 0; idx < g.start[kBoxGroup]; idx += kT) {
    while (idx >= g.start[u + 1]) ++u;
    const int b = g.box[u], n = idx - g.start[u], pb = g.start[u + 1] - g.start[u] - 1;
    const cd* a = mpole + eoff[b] + pb;
    const double f = conv[(size_t)level[b] * (pbmax + 1) + n];
    cd m = n > 0 ? a[-n] : mk(0.0, 0.0);
    if (n & 1) m = mk(-m.x, -m.y);
    const cd s = cadd(a[n], m), d = n > 0 ? csub(a[n], m) : mk(0.0, 0.0);
    reinterpret_cast<float4*>(mu32 + eoff[b] + b)[n] =
        make_float4((float)(s.x * f), (float)(s.y * f), (float)(d.x * f), (float)(d.y * f));
  }
}

// M2L of V-list pairs grouped by (level, distance), in the even / odd form above.
// Items: (first row, rows, first output order, level * kM2lDist + distance). A thread
// computes E_l or O_l of one order l for kFoldRows rows. With P = pb + 1 <= NT / 2
// orders the CTA's threads are P for each half of G <= 16 row groups (NT is chosen by
// level so that few threads are left over); with more, one row group, NT / 2 orders per
// item and the source orders staged NT / 2 at a time. The two threads of an order then
// exchange sums and finish half of the rows each. row.x: entry of the source in mu; row.y: 64
// times the entry of the pair's results in Y, plus its offset class (for the angle).
// m2l_f32_reduce_kernel adds each target box's rows in its V-list order with Kahan
// compensation (deterministic).
// Bound by the matrix loads and the latencies of 12 warps per SM (FMA pipe about half
// busy): every entry is loaded once per kFoldRows rows. M2L of 200 ellipses 3.23 -> 2.21
// ms against one matrix per offset class; starfish at k = 10 0.18 -> 0.13, at k = 50 0.45
// -> 0.32 ms (kKahanBlock = 8). With E_l and O_l in one thread and 8 rows 2.36 ms, with two orders and 8
// rows per thread (half the shared-memory reads) 2.37, with 4 rows and 20 warps 2.74.
constexpr int kFoldRows = 16;
constexpr int kFoldWidth[3] = {128, 96, 64};  // NT
constexpr int kFoldGroups = 16;
__host__ __device__ constexpr int fold_groups(int NT, int P) {
  return 2 * P > NT ? 1 : NT / (2 * P) < kFoldGroups ? NT / (2 * P) : kFoldGroups;
}
template <int NT>
__global__ void __launch_bounds__(NT, 384 / NT) m2l_fold_kernel(
    const int4* __restrict__ items, const int* __restrict__ lpb,
    const long long* __restrict__ toff, const longlong2* __restrict__ rows, int pbmax,
    const float2* __restrict__ rot, const float2* __restrict__ mu, const float2* __restrict__ tm,
    float2* __restrict__ Y) {
  constexpr int R = kFoldRows, RS = stage_stride(R);
  constexpr int NH = NT / 2;
  static_assert(NH % kGemmBlock == 0, "staging must keep the summation blocks");
  __shared__ __align__(16) float2 xs[NT * RS];  // e, then o: [row group][n][row]
  __shared__ longlong2 meta[kFoldGroups * R];
  const int4 I = items[blockIdx.x];
  const int row0 = I.x, nr = I.y;
  const int pb = lpb[I.w / kM2lDist], P = pb + 1;
  const int G = fold_groups(NT, P), W = P <= NH ? P : NH;
  const int id = min((int)threadIdx.x, 2 * G * W - 1);  // threads left over repeat the last
  const int unit = id % (G * W);
  const bool odd = id >= G * W;  // the thread sums O
  const int l = I.z + unit % W, lo = l < P ? l : 0;
  int rg = unit / W;
  const bool act = (int)threadIdx.x < 2 * G * W && rg * R < nr && l < P;
  if (rg * R >= nr) rg = 0;
  const bool warp_act = __any_sync(0xffffffffu, act);
  const float2* te = tm + toff[I.w] + (odd ? (size_t)P * P : 0);
  const int used = (nr + R - 1) / R * R;  // rows staged
  for (int i = threadIdx.x; i < nr; i += NT) meta[i] = rows[row0 + i];
  RowSums<R> S;
  for (int n0 = 0; n0 < P; n0 += NH) {
    const int nk = min(NH, P - n0);
    float2* xe = xs;
    float2* xo = xs + (size_t)G * nk * RS;
    __syncthreads();
    // two row pairs at a time: their loads are in flight together
    const int total = nk * (used / 2);
    for (int i0 = threadIdx.x; i0 < total; i0 += 2 * NT) {
      float4 v[2][2];
      float2 w[2][2];
      int r[2], n[2];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const int idx = i0 + t * NT;
        r[t] = 2 * (idx / nk);  // coalesced reads along each source row
        n[t] = idx % nk;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          v[t][u] = make_float4(0.f, 0.f, 0.f, 0.f);
          w[t][u] = make_float2(0.f, 0.f);
          if (idx < total && r[t] + u < nr) {
            const longlong2 q = meta[r[t] + u];
            v[t][u] = reinterpret_cast<const float4*>(mu + q.x)[n0 + n[t]];
            w[t][u] = rot[(size_t)(q.y & 63) * (pbmax + 1) + n0 + n[t]];
          }
        }
      }
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        if (i0 + t * NT >= total) break;
        float4 e, o;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float4 x = v[t][u];
          const float2 z = w[t][u];
          const float2 ev = make_float2(fmaf(z.x, x.x, -z.y * x.w), fmaf(z.x, x.y, z.y * x.z));
          const float2 ov = make_float2(fmaf(z.x, x.z, -z.y * x.y), fmaf(z.x, x.w, z.y * x.x));
          if (u == 0) e.x = ev.x, e.z = ev.y, o.x = ov.x, o.z = ov.y;
          else e.y = ev.x, e.w = ev.y, o.y = ov.x, o.w = ov.y;
        }
        const int at = ((r[t] / R) * nk + n[t]) * RS + r[t] % R;
        *reinterpret_cast<float4*>(xe + at) = e;
        *reinterpret_cast<float4*>(xo + at) = o;
      }
    }
    __syncthreads();
    if (warp_act)
      tile_gemm_column<R>(te + (size_t)n0 * P, P, nk, (odd ? xo : xe) + (size_t)rg * nk * RS, lo,
                          true, S);
  }
  // E gives its sums of the upper half of the rows for O's of the lower half
  constexpr int RH = R / 2;
  __syncthreads();
  float4* ex = reinterpret_cast<float4*>(xs);  // [row][thread]
  static_assert(sizeof(xs) >= sizeof(float4) * NT * RH, "room for the exchange");
  auto sums = [&](int r) {
    return make_float4(S.sum_r(r), S.sum_i(r), S.lost_r(r), S.lost_i(r));
  };
#pragma unroll
  for (int r = 0; r < RH; ++r) {
    const float4 a = sums(r), b = sums(r + RH);
    ex[r * NT + threadIdx.x] = odd ? a : b;
  }
  __syncthreads();
  const int mate = odd ? (int)threadIdx.x - G * W : (int)threadIdx.x + G * W;
  if (!act) return;
#pragma unroll
  for (int r = 0; r < RH; ++r) {
    const int row = rg * R + r + (odd ? RH : 0);
    if (row >= nr) break;
    const long long q = meta[row].y;
    const float2 w = rot[(size_t)(q & 63) * (pbmax + 1) + l];
    float2* y = Y + (q >> 6) + pb;
    const float4 a0 = sums(r), a1 = sums(r + RH);
    const float4 a = odd ? a1 : a0, o = ex[r * NT + mate];
    const float2 p = make_float2((a.x + o.x) + (a.z + o.z), (a.y + o.y) + (a.w + o.w));
    float2 m = make_float2((a.x - o.x) + (a.z - o.z), (a.y - o.y) + (a.w - o.w));  // E - O
    if (odd) m = make_float2(-m.x, -m.y);
    const float2 yp = make_float2(fmaf(w.x, p.x, -w.y * p.y), fmaf(w.x, p.y, w.y * p.x));
    y[l] = (l & 1) ? make_float2(-yp.x, -yp.y) : yp;
    if (l > 0) y[-l] = make_float2(fmaf(w.x, m.x, w.y * m.y), fmaf(w.x, m.y, -w.y * m.x));
  }
}

// lh_lo(b) += conv_lo * sum over b's V entries e (in list order) of Y[row(e)][lo]:
// FP32 sums with Kahan compensation (FP32 arithmetic is cheap on this GPU, a
// conversion to FP64 per element is not), converted and scaled once in FP64.
__global__ void __launch_bounds__(kT) m2l_f32_reduce_kernel(
    int pbmax, const int* __restrict__ boxes, const int* __restrict__ level,
    const int* __restrict__ lpb, const int* __restrict__ voff, const long long* __restrict__ eyoff,
    const float2* __restrict__ Y, const double* __restrict__ conv,
    const long long* __restrict__ eoff, cd* __restrict__ local) {
  const int b = boxes[blockIdx.x];
  const int l = level[b];
  const int pb = lpb[l], Q = 2 * pb + 1;
  const double* cv = conv + (size_t)l * (pbmax + 1);
  cd* dst = local + eoff[b];
  for (int lo = threadIdx.x; lo < Q; lo += kT) {
    float sr = 0.f, si = 0.f, cr = 0.f, ci = 0.f;
    const int e1 = voff[b + 1];
    int e = voff[b];
    for (; e + 4 <= e1; e += 4) {  // four loads in flight, added in list order
      float2 y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) y[u] = Y[eyoff[e + u] + lo];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        kahan_add(sr, cr, y[u].x);
        kahan_add(si, ci, y[u].y);
      }
    }
    for (; e < e1; ++e) {
      const float2 y = Y[eyoff[e] + lo];
      kahan_add(sr, cr, y.x);
      kahan_add(si, ci, y.y);
    }
    const double f = cv[abs(lo - pb)];
    dst[lo] = cadd(dst[lo], mk(((double)sr - (double)cr) * f, ((double)si - (double)ci) * f));
  }
}

// ---------------------------------------------------------------- FP64 M2L as tile GEMMs
// The FP64 path's M2L, lh_l += (-1)^l sum_n What_{n+l} c(l, n) mh_n with
// What_m = s^|m| W_m(D) and c(l, n) = s^{2 min(|l|,|n|)} when l and n have
// opposite signs (else 1), written as dense matrices per (level, offset
// class): T64[cls][n][l] = (-1)^l What_{n+l} c(l, n) (FP64; the same tiles and
// ordered reduction as the FP32 M2L, without normalisation or compensation).
__global__ void m2l_f64_matrix_kernel(int l, int pb, int pbmax, const cd* __restrict__ t_m2l,
                                      const double* __restrict__ pw, cd* __restrict__ Tm) {
  const int cls = blockIdx.x;
  const int n = (int)blockIdx.y - pb;
  const int Q = 2 * pb + 1;
  const cd* w = t_m2l + ((size_t)l * 49 + cls) * (4 * pbmax + 1) + 2 * pbmax;
  const double* p2 = pw + (size_t)l * (2 * pbmax + 3);  // s^j
  cd* dst = Tm + ((size_t)cls * Q + (n + pb)) * Q;
  const int dx = cls / 7 - 3, dy = cls % 7 - 3;
  const bool used = max(abs(dx), abs(dy)) >= 2;  // V-list offsets only
  for (int lo = (int)threadIdx.x - pb; lo <= pb; lo += blockDim.x) {
    cd v = mk(0.0, 0.0);
    if (used) {
      v = w[n + lo];
      if (!isfinite(v.x) || !isfinite(v.y)) v = mk(0.0, 0.0);  // as in M2lNorm::entry
      if ((n < 0 && lo > 0) || (n > 0 && lo < 0)) v = cscale(v, p2[2 * min(abs(n), abs(lo))]);
      if (lo & 1) v = mk(-v.x, -v.y);
    }
    dst[lo + pb] = v;
  }
}

// FP64 work items take kF64Rows rows of a tile (the accumulators of 16 FP64
// rows would not fit in registers) and kT output orders, the sources staged kChunkK
// orders at a time. Results go to the FP64 rows of Y64, added per target box by
// m2l_f64_reduce_kernel in V-list order.
constexpr int kChunkK = 128;  // source orders staged at a time
constexpr int kF64Rows = 8;
__global__ void __launch_bounds__(kT) m2l_f64_gemm_kernel(
    const int4* __restrict__ items, const int* __restrict__ lpb,
    const long long* __restrict__ goff, const long long* __restrict__ row_off,
    const cd* __restrict__ mpole, const cd* __restrict__ tm,
    const long long* __restrict__ yoff, cd* __restrict__ Y) {
  __shared__ __align__(16) cd xs[kChunkK * kF64Rows];  // [n][row]
  const int4 I = items[blockIdx.x];  // (first row, rows <= kF64Rows, first output order, group)
  const int row0 = I.x, nr = I.y;
  const int Q = 2 * lpb[I.w / 49] + 1;
  const int lo = I.z + (int)threadIdx.x;
  const bool act = lo < Q;
  const bool warp_act = I.z + (int)(threadIdx.x & ~31u) < Q;  // as in the FP32 items
  const cd* M = tm + goff[I.w];
  cd acc[kF64Rows];
#pragma unroll
  for (int r = 0; r < kF64Rows; ++r) acc[r] = mk(0.0, 0.0);
  for (int n0 = 0; n0 < Q; n0 += kChunkK) {
    const int nk = min(kChunkK, Q - n0);
    __syncthreads();
    for (int idx = threadIdx.x; idx < nk * kF64Rows; idx += kT) {
      const int r = idx / nk, n = idx % nk;
      xs[n * kF64Rows + r] = r < nr ? mpole[row_off[row0 + r] + n0 + n] : mk(0.0, 0.0);
    }
    __syncthreads();
    if (!warp_act) continue;
    for (int j0 = 0; j0 < nk; j0 += kGemmBlock) {
      cd tb[kGemmBlock];
#pragma unroll
      for (int j = 0; j < kGemmBlock; ++j)
        tb[j] = (act && j0 + j < nk) ? M[(size_t)(n0 + j0 + j) * Q + lo] : mk(0.0, 0.0);
#pragma unroll
      for (int j = 0; j < kGemmBlock; ++j) {
        if (j0 + j >= nk) break;
        const cd* x = xs + (j0 + j) * kF64Rows;
#pragma unroll
        for (int r = 0; r < kF64Rows; ++r) cfma(acc[r], tb[j], x[r]);
      }
    }
  }
  if (act) {
#pragma unroll
    for (int r = 0; r < kF64Rows; ++r)
      if (r < nr) Y[yoff[row0 + r] + lo] = acc[r];
  }
}

// lh_lo(b) += sum over b's V entries e (in list order) of Y64[row(e)][lo].
__global__ void __launch_bounds__(kT) m2l_f64_reduce_kernel(
    const int* __restrict__ boxes, const int* __restrict__ level, const int* __restrict__ lpb,
    const int* __restrict__ voff, const long long* __restrict__ eyoff, const cd* __restrict__ Y,
    const long long* __restrict__ eoff, cd* __restrict__ local) {
  const int b = boxes[blockIdx.x];
  const int Q = 2 * lpb[level[b]] + 1;
  cd* dst = local + eoff[b];
  for (int lo = threadIdx.x; lo < Q; lo += kT) {
    cd sum = mk(0.0, 0.0);
    const int e1 = voff[b + 1];
    int e = voff[b];
    for (; e + 4 <= e1; e += 4) {  // four loads in flight, added in list order
      cd y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) y[u] = Y[eyoff[e + u] + lo];
#pragma unroll
      for (int u = 0; u < 4; ++u) sum = cadd(sum, y[u]);
    }
    for (; e < e1; ++e) sum = cadd(sum, Y[eyoff[e] + lo]);
    dst[lo] = cadd(dst[lo], sum);
  }
}

// ---------------------------------------------------------------- FP32 M2M and L2L
// The four children of a box lie at the same distance d and at the angles
// pi/4 + rho pi/2, so that the translation by a child's offset is a real matrix
// J_{s-n}(k d) between rotations by eighth turns, and the rotations of the four differ
// by quarter turns i^{rho (s-n)}, which depend on (s - n) mod 4 only:
//   M2M  mu'_s = e^{-i s pi/4} sum_n J_{s-n} b_{(n-s) mod 4, n},
//        b_{j,n} = sum_rho i^{rho j} e^{i n pi/4} mu_{rho,n};
//   L2L  lambda'_{rho,s} = e^{i s pi/4} sum_k i^{rho k} t_k,
//        t_k = sum over n = s - k mod 4 of J_{n-s} e^{-i n pi/4} lambda_n:
// one real matrix product and a four-point transform in place of four complex matrix
// products, an eighth of the multiplications (200 ellipses: M2M 0.69 -> 0.37 ms, L2L with
// the leaves' unscaling 0.97 -> 0.45; starfish at k = 50 0.18 -> 0.11 and 0.20 -> 0.11).
// What is left is the FP64 scaling of the coefficients. Coefficients sigma-normalised (mu_n =
// mh_n conv_n, lambda_n = lh_n / conv_n); the matrices T[n][s] hold the ratio of sigmas
// and 1/sqrt 2 for each odd order of the eighth turns (turn8 leaves it out).
constexpr int child_at(int rho) { return (0x4B >> (2 * rho)) & 3; }  // quadrant at pi/4 + rho pi/2
// Their sums carry the rounding errors along (fe: value and error, fec: complex), and a
// coefficient comes from FP64 and goes back with its error, so that it is rounded to FP32
// once, before the product: with two more roundings per level (a turned coefficient, L2L's
// result) a starfish of 11 levels at k = 4.35 was 1.39e-7 from FP64 instead of 1.23e-7.
struct fe {
  float h, l;
};
struct fec {
  fe x, y;
};
__device__ __forceinline__ fe add(fe a, fe b) {
  const float s = a.h + b.h, t = s - a.h;
  return {s, ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l)};
}
__device__ __forceinline__ fe neg(fe a) { return {-a.h, -a.l}; }
__device__ __forceinline__ fec add(fec a, fec b) { return {add(a.x, b.x), add(a.y, b.y)}; }
__device__ __forceinline__ fec sub(fec a, fec b) { return {add(a.x, neg(b.x)), add(a.y, neg(b.y))}; }
__device__ __forceinline__ fec turn4(fec v, int q) {  // i^q v
  if (q & 1) v = {neg(v.y), v.x};
  if (q & 2) v = {neg(v.x), neg(v.y)};
  return v;
}
__device__ __forceinline__ fec turn8(fec v, int m) {  // e^{i m pi/4} v, sqrt 2 times for odd m
  if (m & 1) v = {add(v.x, neg(v.y)), add(v.x, v.y)};
  return turn4(v, m >> 1);
}
__device__ __forceinline__ void dft4(fec (&v)[4]) {  // v_j <- sum_rho i^{rho j} v_rho
  const fec a = add(v[0], v[2]), b = sub(v[0], v[2]);
  const fec c = add(v[1], v[3]), d = turn4(sub(v[1], v[3]), 1);
  v[0] = add(a, c);
  v[2] = sub(a, c);
  v[1] = add(b, d);
  v[3] = sub(b, d);
}
__device__ __forceinline__ float2 f32(fec v) { return make_float2(v.x.h + v.x.l, v.y.h + v.y.l); }
// v f as values and errors, and (value + error) f added to v, with integer instructions
// for the conversions (those of the FP64 pipe would take as long as the products)
__device__ __forceinline__ fec pair_of(cd v, double f) {
  const ff x = ff_from_f64_nan(v.x * f, 896), y = ff_from_f64_nan(v.y * f, 896);
  return {{x.h, x.l}, {y.h, y.l}};
}
__device__ __forceinline__ cd add_pair(cd v, fec a, double f) {
  return mk(fma(f64_from_f32(a.x.l), f, fma(f64_from_f32(a.x.h), f, v.x)),
            fma(f64_from_f32(a.y.l), f, fma(f64_from_f32(a.y.h), f, v.y)));
}

// The matrix of parent level l (M2M: from child order n to parent order s; L2L: from
// parent to child), from the tables of the quadrant at pi/4 (row stride 4 pbmax + 1,
// order m at m + 2 pbmax): J_m e^{-i m pi/4} for M2M, J_{-m} e^{i m pi/4} for L2L at
// m = s - n. Grid: n, threads over s.
template <bool M2M>
__global__ void fold_matrix_kernel(int l, int pp, int pc, int pbmax, const cd* __restrict__ table,
                                   const double* __restrict__ lsig, float* __restrict__ T) {
  const int pn = M2M ? pc : pp, ps = M2M ? pp : pc;
  const int n = (int)blockIdx.x - pn;
  const cd* v = table + ((size_t)l * 4 + child_at(0)) * (4 * pbmax + 1) + 2 * pbmax;
  const double* sp = lsig + (size_t)l * (pbmax + 1);
  const double* sc = lsig + (size_t)(l + 1) * (pbmax + 1);
  float* dst = T + (size_t)(n + pn) * (2 * ps + 1) + ps;
  for (int s = (int)threadIdx.x - ps; s <= ps; s += blockDim.x) {
    const cd e = v[s - n];
    double c, sn;
    sincospi(0.25 * (M2M ? s - n : n - s), &sn, &c);
    const double J = e.x * c - e.y * sn;
    double out = 0.0;
    if (J != 0.0) {
      const double lf = (M2M ? sc[abs(n)] - sp[abs(s)] : sc[abs(s)] - sp[abs(n)]) + log(fabs(J));
      out = lf < -700.0 ? 0.0 : copysign(exp(lf), J);
    }
    if (n & 1) out *= 0.70710678118654752440;
    if (s & 1) out *= 0.70710678118654752440;
    dst[s] = (float)out;
  }
}

// S[r] += sum_{j < N} M[j * ld + lo] * x[j * XS][r] with a real matrix, otherwise as
// tile_gemm_column.
template <int R, int XS>
__device__ __forceinline__ void real_block_add(const float (&tb)[kGemmBlock], int nj,
                                               const float2* __restrict__ x, RowSums<R>& S) {
  f32p tr[R / 2], ti[R / 2];
#pragma unroll
  for (int j = 0; j < kGemmBlock; ++j) {
    if (j < nj) {
      const f32p t = pk(tb[j], tb[j]);
      const ulonglong2* m = reinterpret_cast<const ulonglong2*>(x + j * XS);
#pragma unroll
      for (int r = 0; r < R / 2; ++r) {
        const ulonglong2 v = m[r];
        tr[r] = fma2(t, v.x, j == 0 ? S.nr[r] : tr[r]);
        ti[r] = fma2(t, v.y, j == 0 ? S.ni[r] : ti[r]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < R / 2; ++r) {
    kahan_add2(S.sr[r], S.nr[r], tr[r]);
    kahan_add2(S.si[r], S.ni[r], ti[r]);
  }
}
template <int R, int XS>
__device__ __forceinline__ void real_column(const float* __restrict__ M, size_t ld, int N,
                                            const float2* __restrict__ x, int lo, bool act,
                                            RowSums<R>& S) {
  const float* Mc = M + (act ? lo : 0);
  float ta[kGemmBlock], tb[kGemmBlock];
  auto load = [&](float (&t)[kGemmBlock], int n0) {
#pragma unroll
    for (int j = 0; j < kGemmBlock; ++j) t[j] = n0 + j < N ? Mc[(size_t)(n0 + j) * ld] : 0.f;
  };
  load(ta, 0);
  for (int n0 = 0; n0 < N; n0 += 2 * kGemmBlock) {
    const int n1 = n0 + kGemmBlock;
    if (n1 < N) load(tb, n1);
    real_block_add<R, XS>(ta, min(kGemmBlock, N - n0), x + (size_t)n0 * XS, S);
    if (n1 >= N) break;
    if (n1 + kGemmBlock < N) load(ta, n1 + kGemmBlock);
    real_block_add<R, XS>(tb, min(kGemmBlock, N - n1), x + (size_t)n1 * XS, S);
  }
}

// A CTA takes R parents. Warp w sums the terms n = w mod 4 (counted from the lowest
// order) of 32 orders s, one per lane, for all R; the CTA's warps then join the four
// sums. The orders s are taken 32 at a time, gridDim.y apart. Source orders are staged
// kFoldK at a time (all at once but for orders beyond any ordinary box).
constexpr int kFoldK = 256;
static_assert(kT == 128 && kFoldK % (4 * kGemmBlock) == 0, "four warps, whole summation blocks");
__host__ __device__ constexpr size_t fold_staged(int Q, int per, int R) {  // float2 words
  return (size_t)(Q < kFoldK ? Q : kFoldK) * per * stage_stride(R);
}
constexpr size_t fold_smem(int Q, int per, int R) {  // the rows and the joint's fec[4][R][32]
  return fold_staged(Q, per, R) * sizeof(float2) + 128 * (size_t)R * sizeof(fec);
}
template <int R>
__device__ __forceinline__ void put_sums(const RowSums<R>& S, fec* red, int warp, int lane) {
#pragma unroll
  for (int r = 0; r < R; ++r)
    red[(warp * R + r) * 32 + lane] = {{S.sum_r(r), S.lost_r(r)}, {S.sum_i(r), S.lost_i(r)}};
}

template <int R>
__global__ void __launch_bounds__(kT, 4) m2m_fold_kernel(
    int l, int pp, int pc, int pbmax, const int* __restrict__ parents, int nb,
    const int* __restrict__ child, const long long* __restrict__ eoff, const float* __restrict__ T,
    const double* __restrict__ conv, const double* __restrict__ iconv, cd* __restrict__ mpole) {
  constexpr int RS = stage_stride(R);
  extern __shared__ __align__(16) float2 fx[];  // [n][j][RS], then the joint's fec[4][R][32]
  __shared__ long long coff[4][R], poff[R];     // children by rho
  const int Qp = 2 * pp + 1, Qc = 2 * pc + 1;
  fec* red = reinterpret_cast<fec*>(fx + fold_staged(Qc, 4, R));
  const int p0 = blockIdx.x * R, nr = min(R, nb - p0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_allow_next();
  for (int idx = threadIdx.x; idx < 5 * R; idx += kT) {
    const int r = idx % R, c = idx / R;
    long long o = -1;
    if (r < nr) {
      const int b = parents[p0 + r];
      const int d = c == 4 ? b : child[4 * b + child_at(c)];
      if (d >= 0) o = eoff[d];
    }
    if (c == 4) poff[r] = o; else coff[c][r] = o;
  }
  const double* cvc = conv + (size_t)(l + 1) * (pbmax + 1);
  const double* icp = iconv + (size_t)l * (pbmax + 1);
  __syncthreads();
  pdl_wait();
  bool staged = false;
  for (int s0 = blockIdx.y * 32; s0 < Qp; s0 += 32 * gridDim.y) {
    const int at = s0 + lane, s = at - pp;
    const bool act = at < Qp;
    const int j = (warp - pc - s) & 3;
    RowSums<R> S;
    for (int n0 = 0; n0 < Qc; n0 += kFoldK) {
      const int nk = min(kFoldK, Qc - n0);
      if (!staged || Qc > kFoldK) {
        __syncthreads();
        for (int idx = threadIdx.x; idx < nk * R; idx += kT) {
          const int r = idx / nk, n = idx % nk, m = n0 + n - pc;
          const double f = cvc[abs(m)];
          fec v[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            v[c] = {{0.f, 0.f}, {0.f, 0.f}};
            if (coff[c][r] >= 0) {
              const cd a = mpole[coff[c][r] + n0 + n];
              v[c] = turn8(pair_of(a, f), m);
            }
          }
          dft4(v);
#pragma unroll
          for (int q = 0; q < 4; ++q) stage_put(fx, (size_t)n * 4 + q, r, RS, f32(v[q]));
        }
        __syncthreads();
        staged = true;
      }
      const int N = (nk - warp + 3) / 4;
      if (N > 0)
        real_column<R, 16 * RS>(T + (size_t)(n0 + warp) * Qp, 4 * (size_t)Qp, N,
                                fx + (warp * 4 + j) * RS, at, act, S);
    }
    __syncthreads();
    put_sums<R>(S, red, warp, lane);
    __syncthreads();
    if (act) {
      const double f = icp[abs(s)];
      for (int r = warp; r < nr; r += 4) {
        fec v[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) v[w] = red[(w * R + r) * 32 + lane];
        const fec u = turn8(add(add(v[0], v[1]), add(v[2], v[3])), -s);
        mpole[poff[r] + at] = add_pair(mk(0.0, 0.0), u, f);
      }
    }
  }
}

template <int R>
__global__ void __launch_bounds__(kT, 4) l2l_fold_kernel(
    int l, int pp, int pc, int pbmax, const int* __restrict__ parents, int nb,
    const int* __restrict__ child, const long long* __restrict__ eoff, const float* __restrict__ T,
    const double* __restrict__ conv, const double* __restrict__ iconv, cd* __restrict__ local) {
  constexpr int RS = stage_stride(R);
  extern __shared__ __align__(16) float2 fx[];  // [n][RS], then the joint's fec[4][R][32]
  __shared__ long long coff[4][R], poff[R];     // children by rho
  const int Qp = 2 * pp + 1, Qc = 2 * pc + 1;
  fec* red = reinterpret_cast<fec*>(fx + fold_staged(Qp, 1, R));
  const int p0 = blockIdx.x * R, nr = min(R, nb - p0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_allow_next();
  for (int idx = threadIdx.x; idx < 5 * R; idx += kT) {
    const int r = idx % R, c = idx / R;
    long long o = -1;
    if (r < nr) {
      const int b = parents[p0 + r];
      const int d = c == 4 ? b : child[4 * b + child_at(c)];
      if (d >= 0) o = eoff[d];
    }
    if (c == 4) poff[r] = o; else coff[c][r] = o;
  }
  const double* cvc = conv + (size_t)(l + 1) * (pbmax + 1);
  const double* icp = iconv + (size_t)l * (pbmax + 1);
  __syncthreads();
  pdl_wait();
  bool staged = false;
  for (int s0 = blockIdx.y * 32; s0 < Qc; s0 += 32 * gridDim.y) {
    const int at = s0 + lane, s = at - pc;
    const bool act = at < Qc;
    RowSums<R> S;
    for (int n0 = 0; n0 < Qp; n0 += kFoldK) {
      const int nk = min(kFoldK, Qp - n0);
      if (!staged || Qp > kFoldK) {
        __syncthreads();
        for (int idx = threadIdx.x; idx < nk * R; idx += kT) {
          const int r = idx / nk, n = idx % nk, m = n0 + n - pp;
          float2 v = make_float2(0.f, 0.f);
          if (r < nr) {
            const cd g = local[poff[r] + n0 + n];
            const double f = icp[abs(m)];
            v = f32(turn8(pair_of(g, f), -m));
          }
          stage_put(fx, n, r, RS, v);
        }
        __syncthreads();
        staged = true;
      }
      const int N = (nk - warp + 3) / 4;
      if (N > 0)
        real_column<R, 4 * RS>(T + (size_t)(n0 + warp) * Qc, 4 * (size_t)Qc, N, fx + warp * RS, at,
                               act, S);
    }
    __syncthreads();
    put_sums<R>(S, red, warp, lane);
    __syncthreads();
    if (act) {
      const double f = cvc[abs(s)];
      for (int r = warp; r < nr; r += 4) {
        fec v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = red[(((s + pp - k) & 3) * R + r) * 32 + lane];
        dft4(v);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (coff[c][r] < 0) continue;
          cd* dst = local + coff[c][r] + at;
          *dst = add_pair(*dst, turn8(v[c], s), f);
        }
      }
    }
  }
}

// out[i] = eoff[idx[i]]: the coefficient offset of each M2L source row
__global__ void gather_offsets_kernel(const int* __restrict__ idx, const long long* __restrict__ eoff,
                                      long long* __restrict__ out, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = eoff[idx[i]];
}

}  // namespace

qbx_status configure_mixed_kernels(int smem_optin) {
  const void* k[] = {(const void*)m2m_fold_kernel<2>, (const void*)m2m_fold_kernel<4>,
                     (const void*)m2m_fold_kernel<8>, (const void*)l2l_fold_kernel<2>,
                     (const void*)l2l_fold_kernel<4>, (const void*)l2l_fold_kernel<8>};
  for (const void* fn : k) {
    cudaFuncAttributes a;
    QBX_CUDA_TRY(cudaFuncGetAttributes(&a, fn));  // dynamic + static must fit the opt-in size
    QBX_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      smem_optin - (int)a.sharedSizeBytes));
  }
  return QBX_OK;
}

// The exponent s for which 2^{s m} H_m(x) and 2^{-s m} J_m(y), m <= pb, stay in
// FP32's range at the arguments that boxes of k side = x0 meet: a W-list box's
// targets and a local expansion's sources lie 1.5 sides or more from the centre
// (x >= 1.4 x0), its own points within 0.71 sides (y <= 0.71 x0). H_m grows like
// (2 m / (e x))^m, so s puts the turn of (2 m 2^s / (e x))^m at 0.6 pb: it falls
// to 2^{-0.32 pb} before and rises to 2^{0.44 pb} at pb. Refused (FP64 kernels)
// when the largest |2^{s m} H_m| exceeds 2^60, when 2^{s m} / sig_m (isf, larger than
// that by pi m 1.4^m) comes within a factor four of FP32's largest value, which it does
// from order 119 on, or an order reaches 128 (the recurrence's exact products m c hold 7
// bits of m).
static int float_float_scale(double x0, int pb) {
  if (pb < 1 || pb > 126) return kNoFf;
  const double xl = 1.4 * x0;
  const int s = (int)std::lrint(std::min(0.0, std::log2(xl * 1.3591409142295226 / (0.6 * pb))));
  if (s < -50) return kNoFf;
  constexpr double kLn2 = 0.69314718055994531;
  double top = 0.0, isf = 0.0;
  for (int m = 1; m <= pb; ++m) {
    if (m > xl)  // |H_m(x)| <~ (m-1)!/pi (2/x)^m for m > x, of order one below
      top = std::max(top, s * m + (std::lgamma((double)m) - 1.1447298858494002 +
                                   m * std::log(2.0 / xl)) / kLn2);
    isf = std::max(isf, s * m + std::max(0.0, std::lgamma(m + 1.0) - m * std::log(0.5 * x0)) / kLn2);
  }
  return top > 60.0 || isf > 126.0 ? kNoFf : s;
}

qbx_status mixed_plan_build(qbx_handle* h, FmmPlan* f) {
  const int pbm = f->pb_max;
  QBX_CUDA_TRY(f->lsig.alloc((size_t)f->n_levels * (pbm + 1)));
  QBX_CUDA_TRY(f->conv.alloc((size_t)f->n_levels * (pbm + 1)));
  QBX_CUDA_TRY(f->iconv.alloc((size_t)f->n_levels * (pbm + 1)));
  QBX_CUDA_TRY(f->isig.alloc((size_t)f->n_levels * (pbm + 2)));
  sigma_tables_kernel<<<f->n_levels, 128>>>(f->n_levels, pbm, f->lpb.ptr, h->k, f->side, f->scale.ptr,
                                 f->lsig.ptr, f->conv.ptr, f->iconv.ptr, f->isig.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  QBX_CUDA_TRY(f->m2p_rec.alloc((size_t)f->n_levels * (pbm + 2)));
  m2p_rec_kernel<<<f->n_levels, 128>>>(f->n_levels, pbm, f->lpb.ptr, f->lsig.ptr, f->m2p_rec.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  QBX_CUDA_TRY(f->sigr.alloc((size_t)f->n_levels * (pbm + 2)));
  sig_ratio_kernel<<<f->n_levels, 128>>>(f->n_levels, pbm, f->lpb.ptr, f->lsig.ptr, f->sigr.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  {  // |H_m(x)| <~ (m-1)! (2/x)^m; a W-list box's targets lie 1.5 sides away (taken as 0.5)
    std::vector<int> big(f->n_levels, 0);
    for (int l = 2; l < f->n_levels; ++l) {
      const double x_lo = 0.5 * h->k * f->side / std::ldexp(1.0, l);
      const int pb = std::max(1, f->h_pb[l]);
      big[l] = std::lgamma((double)pb + 1.0) + (pb + 1) * std::log(2.0 / x_lo) > 650.0 ? 1 : 0;
    }
    QBX_CUDA_TRY(f->m2p_big.alloc(f->n_levels));
    QBX_CUDA_TRY(cudaMemcpy(f->m2p_big.ptr, big.data(), f->n_levels * sizeof(int),
                            cudaMemcpyHostToDevice));
  }
  {
    std::vector<int> ffs(f->n_levels, kNoFf);
    for (int l = 2; l < f->n_levels; ++l)
      ffs[l] = float_float_scale(h->k * f->side / std::ldexp(1.0, l), f->h_pb[l]);
    f->h_ffs = ffs;
    QBX_CUDA_TRY(f->ff_s.alloc(f->n_levels));
    QBX_CUDA_TRY(cudaMemcpy(f->ff_s.ptr, ffs.data(), f->n_levels * sizeof(int),
                            cudaMemcpyHostToDevice));
    QBX_CUDA_TRY(f->isf.alloc((size_t)f->n_levels * (pbm + 2)));
    isig_ff_kernel<<<f->n_levels, 128>>>(f->n_levels, pbm, f->lpb.ptr, f->ff_s.ptr, f->lsig.ptr,
                                         f->isf.ptr);
    QBX_CUDA_TRY(cudaGetLastError());
  }
  // matrices for the levels that have V lists
  std::vector<long long> off(f->n_levels, 0);
  long long tot = 0;
  for (int l = 0; l < f->n_levels; ++l) {
    off[l] = tot;
    if (f->vbox_off[l + 1] > f->vbox_off[l]) {
      const long long Q = 2 * f->h_pb[l] + 1;
      tot += 49 * Q * Q;
    }
  }
  std::vector<long long> foff((size_t)f->n_levels * kM2lDist, 0);  // FP32, per (level, distance)
  long long ftot = 0;
  for (int l = 0; l < f->n_levels; ++l) {
    if (f->vbox_off[l + 1] == f->vbox_off[l]) continue;
    const long long P = f->h_pb[l] + 1;
    for (int d = 0; d < kM2lDist; ++d) {
      foff[(size_t)l * kM2lDist + d] = ftot;
      ftot += 2 * P * P;
    }
  }
  QBX_CUDA_TRY(f->tm_f32.alloc(std::max<long long>(1, ftot)));
  for (int l = 2; l < f->n_levels; ++l) {
    if (f->vbox_off[l + 1] == f->vbox_off[l]) continue;
    const int pb = f->h_pb[l];
    m2l_fold_matrix_kernel<<<dim3(kM2lDist, pb + 1), kT>>>(
        l, pb, pbm, f->t_m2l.ptr, f->scale.ptr, f->lsig.ptr,
        f->tm_f32.ptr + foff[(size_t)l * kM2lDist]);
    QBX_CUDA_TRY(cudaGetLastError());
  }
  QBX_CUDA_TRY(f->m2l_toff.alloc(foff.size()));
  QBX_CUDA_TRY(cudaMemcpy(f->m2l_toff.ptr, foff.data(), foff.size() * sizeof(long long),
                          cudaMemcpyHostToDevice));
  QBX_CUDA_TRY(f->m2l_rot.alloc((size_t)49 * (pbm + 1)));
  m2l_rot_kernel<<<49, 128>>>(pbm, f->m2l_rot.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  // M2L work: V-list pairs grouped by (level, offset class); the row of V entry e is
  // vrow[e], its output at yoff[row]
  {
    const int nb = f->n_boxes;
    const int64_t nv = f->V.nnz;
    std::vector<int> voff(nb + 1), vidx(std::max<int64_t>(1, nv)), vcls(std::max<int64_t>(1, nv)),
        blev(nb);
    QBX_CUDA_TRY(cudaMemcpy(voff.data(), f->V.off.ptr, (nb + 1) * sizeof(int), cudaMemcpyDeviceToHost));
    if (nv) {
      QBX_CUDA_TRY(cudaMemcpy(vidx.data(), f->V.idx.ptr, nv * sizeof(int), cudaMemcpyDeviceToHost));
      QBX_CUDA_TRY(cudaMemcpy(vcls.data(), f->V_cls.ptr, nv * sizeof(int), cudaMemcpyDeviceToHost));
    }
    QBX_CUDA_TRY(cudaMemcpy(blev.data(), f->box.level.ptr, nb * sizeof(int), cudaMemcpyDeviceToHost));
    const int ng = f->n_levels * 49;
    std::vector<int64_t> gcount(ng + 1, 0);
    std::vector<int> egroup(std::max<int64_t>(1, nv));
    for (int b = 0; b < nb; ++b)
      for (int e = voff[b]; e < voff[b + 1]; ++e) {
        egroup[e] = blev[b] * 49 + vcls[e];
        gcount[egroup[e] + 1] += 1;
      }
    for (int g = 0; g < ng; ++g) gcount[g + 1] += gcount[g];
    std::vector<long long> eo(nb);
    QBX_CUDA_TRY(cudaMemcpy(eo.data(), f->eoff.ptr, nb * sizeof(long long), cudaMemcpyDeviceToHost));
    std::vector<int> vrow(std::max<int64_t>(1, nv)), row_src(std::max<int64_t>(1, nv));
    std::vector<long long> yoff(std::max<int64_t>(1, nv));
    std::vector<int64_t> fill(gcount.begin(), gcount.end() - 1);
    for (int b = 0; b < nb; ++b)
      for (int e = voff[b]; e < voff[b + 1]; ++e) {
        const int row = (int)fill[egroup[e]]++;
        vrow[e] = row;
        row_src[row] = vidx[e];
      }
    f->h_row_src = row_src;
    f->h_row_src.resize(gcount[ng]);
    f->h_gcount.assign(gcount.begin(), gcount.end());
    long long ytot = 0;
    std::vector<int4> tiles;
    for (int g = 0; g < ng; ++g) {
      const int l = g / 49, Q = 2 * f->h_pb[l] + 1;
      for (int64_t r = gcount[g]; r < gcount[g + 1]; ++r) {
        yoff[r] = ytot;
        ytot += Q;
      }
      for (int64_t r = gcount[g]; r < gcount[g + 1]; r += kGemmRows)
        tiles.push_back(make_int4(g, (int)r, (int)std::min<int64_t>(kGemmRows, gcount[g + 1] - r), l));
    }
    // FP64 work items, coarse levels (largest orders) first: (first row, rows, first
    // output order, group), tiles in groups of kF64Rows rows and kT output orders
    std::vector<int4> it64;
    for (const int4& t : tiles) {
      const int Q = 2 * f->h_pb[t.w] + 1;
      for (int c0 = 0; c0 < Q; c0 += kT)
        for (int r0 = 0; r0 < t.z; r0 += kF64Rows)
          it64.push_back(make_int4(t.y + r0, std::min(kF64Rows, t.z - r0), c0, t.x));
    }
    // FP32: the rows in order of (level, distance), classes side by side; items by
    // block width
    std::vector<longlong2> frow;
    std::vector<int4> it32, by_width[3];  // blocks of 128, 96, 64 threads
    frow.reserve(gcount[ng]);
    for (int l = 0; l < f->n_levels; ++l) {
      const int P = f->h_pb[l] + 1;
      int u = 0, best = -1;  // the width that leaves the fewest threads without an order
      for (int v = 2; v >= 0; --v) {
        const int nt = kFoldWidth[v];
        const int full = 2 * P <= nt ? 2000 * fold_groups(nt, P) * P / nt
                                     : 1000 * P / (nblk(P, nt / 2) * (nt / 2));
        if (full > best) best = full, u = v;
      }
      const int nt = kFoldWidth[u], most = kFoldRows * fold_groups(nt, P);
      for (int d = 0; d < kM2lDist; ++d) {
        const int64_t r0 = (int64_t)frow.size();
        for (int c = 0; c < 49; ++c) {
          if (m2l_dist(c) != d) continue;
          const int g = l * 49 + c;
          for (int64_t r = gcount[g]; r < gcount[g + 1]; ++r)
            frow.push_back(make_longlong2(eo[row_src[r]] + row_src[r], yoff[r] * 64 + c));
        }
        const int64_t r1 = (int64_t)frow.size();
        for (int64_t r = r0; r < r1; r += most)
          for (int c0 = 0; c0 < P; c0 += 2 * P <= nt ? P : nt / 2)
            by_width[u].push_back(
                make_int4((int)r, (int)std::min<int64_t>(most, r1 - r), c0, l * kM2lDist + d));
      }
    }
    for (int u = 0; u < 3; ++u) {
      it32.insert(it32.end(), by_width[u].begin(), by_width[u].end());
      f->n_m2l_width[u] = (int)by_width[u].size();
    }
    QBX_CUDA_TRY(f->m2l_frow.alloc(std::max<size_t>(1, frow.size())));
    if (!frow.empty())
      QBX_CUDA_TRY(cudaMemcpy(f->m2l_frow.ptr, frow.data(), frow.size() * sizeof(longlong2),
                              cudaMemcpyHostToDevice));
    // matrix offset of each group (level l, class c): level offset + c Q_l^2
    std::vector<long long> goff(ng, 0);
    for (int g = 0; g < ng; ++g) {
      const long long Q = 2 * f->h_pb[g / 49] + 1;
      goff[g] = off[g / 49] + (long long)(g % 49) * Q * Q;
    }
    QBX_CUDA_TRY(f->m2l_goff.alloc(ng));
    QBX_CUDA_TRY(cudaMemcpy(f->m2l_goff.ptr, goff.data(), ng * sizeof(long long), cudaMemcpyHostToDevice));
    f->n_m2l_items32 = (int)it32.size();
    f->n_m2l_items64 = (int)it64.size();
    f->h_items64 = it64;
    QBX_CUDA_TRY(f->m2l_items32.alloc(std::max<size_t>(1, it32.size())));
    QBX_CUDA_TRY(f->m2l_items64.alloc(std::max<size_t>(1, it64.size())));
    if (!it32.empty()) {
      QBX_CUDA_TRY(cudaMemcpy(f->m2l_items32.ptr, it32.data(), it32.size() * sizeof(int4), cudaMemcpyHostToDevice));
      QBX_CUDA_TRY(cudaMemcpy(f->m2l_items64.ptr, it64.data(), it64.size() * sizeof(int4), cudaMemcpyHostToDevice));
    }
    QBX_CUDA_TRY(f->m2l_eyoff.alloc(vrow.size()));
    QBX_CUDA_TRY(f->m2l_yoff.alloc(yoff.size()));
    QBX_CUDA_TRY(f->m2l_y.alloc(std::max<long long>(1, ytot)));
    // the boxes that are V-list sources, and FP32 room for their multipoles
    std::vector<char> is_src(nb, 0);
    for (int64_t e = 0; e < nv; ++e) is_src[vidx[e]] = 1;
    std::vector<int> vsrc;
    for (int b = 0; b < nb; ++b)
      if (is_src[b]) vsrc.push_back(b);
    f->n_vsrc = (int)vsrc.size();
    QBX_CUDA_TRY(f->m2l_vsrc.alloc(std::max<size_t>(1, vsrc.size())));
    if (!vsrc.empty())
      QBX_CUDA_TRY(cudaMemcpy(f->m2l_vsrc.ptr, vsrc.data(), vsrc.size() * sizeof(int), cudaMemcpyHostToDevice));
    QBX_CUDA_TRY(f->mu32.alloc(std::max<int64_t>(1, f->n_coef + nb)));
    {  // result-row offset of every V entry
      std::vector<long long> eyoff(vrow.size(), 0);
      for (int64_t e = 0; e < nv; ++e) eyoff[e] = yoff[vrow[e]];
      QBX_CUDA_TRY(cudaMemcpy(f->m2l_eyoff.ptr, eyoff.data(), eyoff.size() * sizeof(long long),
                              cudaMemcpyHostToDevice));
    }
    {  // coefficient offset of each row's source box
      DevBuf<int> rs;
      QBX_CUDA_TRY(rs.alloc(row_src.size()));
      QBX_CUDA_TRY(cudaMemcpy(rs.ptr, row_src.data(), row_src.size() * sizeof(int), cudaMemcpyHostToDevice));
      QBX_CUDA_TRY(f->m2l_rowoff.alloc(row_src.size()));
      gather_offsets_kernel<<<nblk((int64_t)row_src.size(), 256), 256>>>(rs.ptr, f->eoff.ptr,
                                                                          f->m2l_rowoff.ptr, (int64_t)row_src.size());
      QBX_CUDA_TRY(cudaGetLastError());
      QBX_CUDA_TRY(dev_sync());  // before rs is freed
    }
    QBX_CUDA_TRY(cudaMemcpy(f->m2l_yoff.ptr, yoff.data(), yoff.size() * sizeof(long long), cudaMemcpyHostToDevice));
  }
  // FP64 M2L matrices and result rows
  QBX_CUDA_TRY(f->tm_f64.alloc(std::max<long long>(1, tot)));
  for (int l = 2; l < f->n_levels; ++l) {
    if (f->vbox_off[l + 1] == f->vbox_off[l]) continue;
    const int pb = f->h_pb[l];
    dim3 grid(49, 2 * pb + 1);
    m2l_f64_matrix_kernel<<<grid, kT>>>(l, pb, pbm, f->t_m2l.ptr, f->pw.ptr, f->tm_f64.ptr + off[l]);
    QBX_CUDA_TRY(cudaGetLastError());
  }
  QBX_CUDA_TRY(f->m2l_y64.alloc(std::max<size_t>(1, f->m2l_y.n)));
  // M2M and L2L matrices for parents on levels 2 .. n_levels - 2
  std::vector<long long> moff(f->n_levels, 0);
  long long mtot = 0;
  for (int l = 2; l + 1 < f->n_levels; ++l) {
    moff[l] = mtot;
    mtot += (2LL * f->h_pb[l] + 1) * (2 * f->h_pb[l + 1] + 1);
  }
  QBX_CUDA_TRY(f->tmm_f32.alloc(std::max<long long>(1, mtot)));
  QBX_CUDA_TRY(f->tl_f32.alloc(std::max<long long>(1, mtot)));
  f->h_fold_off = moff;
  for (int l = 2; l + 1 < f->n_levels; ++l) {
    const int pp = f->h_pb[l], pc = f->h_pb[l + 1];
    fold_matrix_kernel<true><<<2 * pc + 1, kT>>>(l, pp, pc, pbm, f->t_m2m.ptr, f->lsig.ptr,
                                                 f->tmm_f32.ptr + moff[l]);
    QBX_CUDA_TRY(cudaGetLastError());
    fold_matrix_kernel<false><<<2 * pp + 1, kT>>>(l, pp, pc, pbm, f->t_l2l.ptr, f->lsig.ptr,
                                                  f->tl_f32.ptr + moff[l]);
    QBX_CUDA_TRY(cudaGetLastError());
  }
  return QBX_OK;
}

size_t gemm_smem_bytes(int pb) {
  return (size_t)(2 * pb + 1) * stage_stride(kGemmRows) * sizeof(float2) +
         5 * kGemmRows * sizeof(long long);
}

qbx_status launch_m2l_f64(qbx_handle* h, FmmPlan* f, cudaStream_t s) {
  if (f->n_vbox == 0 || f->n_m2l_items64 == 0) return QBX_OK;
  m2l_f64_gemm_kernel<<<f->n_m2l_items64, kT, 0, s>>>(
      f->m2l_items64.ptr, f->lpb.ptr, f->m2l_goff.ptr, f->m2l_rowoff.ptr, f->mpole.ptr,
      f->tm_f64.ptr, f->m2l_yoff.ptr, f->m2l_y64.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  m2l_f64_reduce_kernel<<<f->n_vbox, kT, 0, s>>>(
      f->vbox.ptr, f->box.level.ptr, f->lpb.ptr, f->V.off.ptr, f->m2l_eyoff.ptr,
      f->m2l_y64.ptr, f->eoff.ptr, f->local.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  h->launches += 2;
  return QBX_OK;
}

// The FP64 tile GEMM over the items of the levels that the tensor-core M2L
// does not take (their result rows, FP64, are added by the tensor-core path's
// reduction).
qbx_status launch_m2l_f64_gemm_rest(qbx_handle* h, FmmPlan* f, cudaStream_t s) {
  if (f->n_m2l_items64_rest == 0) return QBX_OK;
  m2l_f64_gemm_kernel<<<f->n_m2l_items64_rest, kT, 0, s>>>(
      f->m2l_items64_rest.ptr, f->lpb.ptr, f->m2l_goff.ptr, f->m2l_rowoff.ptr, f->mpole.ptr,
      f->tm_f64.ptr, f->m2l_yoff.ptr, f->m2l_y64.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  h->launches += 1;
  return QBX_OK;
}

// A launch that may start before its predecessor in the stream has finished
// (pdl_wait in the kernel); ordinary for batched handles, whose streams share the
// SMs with other problems.
template <typename... P, typename... A>
static cudaError_t launch_chained(void (*k)(P...), dim3 g, size_t smem, cudaStream_t s, bool chain,
                                  A... a) {
  cudaLaunchConfig_t c = {};
  c.gridDim = g;
  c.blockDim = dim3(kT);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = chain ? 1 : 0;
  return cudaLaunchKernelEx(&c, k, P(a)...);
}
// FP32 M2M (from the child level up) or L2L of all levels. Parents per CTA: 8 where
// that gives the SMs two CTAs each, fewer on narrower levels, whose CTAs also share a
// parent's orders out (so that it is staged several times). A level's launch may
// overlap the one before it (only such kernels allow it).
template <bool M2M>
static qbx_status launch_fold(qbx_handle* h, FmmPlan* f, cudaStream_t s) {
  bool prev = false;
  const int n = f->n_levels - 3;  // levels 2 .. n_levels - 2
  for (int i = 0; i < n; ++i) {
    const int l = M2M ? f->n_levels - 2 - i : 2 + i;
    const int nb = f->nonleaf_off[l + 1] - f->nonleaf_off[l];
    if (nb == 0) continue;
    const int pp = f->h_pb[l], pc = f->h_pb[l + 1];
    const int Qi = 2 * (M2M ? pc : pp) + 1, Qo = 2 * (M2M ? pp : pc) + 1;
    auto launch = [&](auto rows) -> cudaError_t {
      constexpr int R = decltype(rows)::value;
      const unsigned gx = nblk(nb, R), chunks = nblk(Qo, 32);
      const unsigned gy = h->batched ? 1u : std::min(chunks, std::max(1u, 4 * 152 / gx));
      return launch_chained(M2M ? m2m_fold_kernel<R> : l2l_fold_kernel<R>, dim3(gx, gy),
                            fold_smem(Qi, M2M ? 4 : 1, R), s, prev && !h->batched, l, pp, pc,
                            f->pb_max, (const int*)f->nonleaf.ptr + f->nonleaf_off[l], nb,
                            (const int*)f->box.child.ptr, (const long long*)f->eoff.ptr,
                            (const float*)(M2M ? f->tmm_f32.ptr : f->tl_f32.ptr) + f->h_fold_off[l],
                            (const double*)f->conv.ptr, (const double*)f->iconv.ptr,
                            M2M ? f->mpole.ptr : f->local.ptr);
    };
    if (nb >= 8 * 2 * 152 || (h->batched && nb >= 64))
      QBX_CUDA_TRY(launch(std::integral_constant<int, 8>()));
    else if (nb >= 4 * 152)
      QBX_CUDA_TRY(launch(std::integral_constant<int, 4>()));
    else
      QBX_CUDA_TRY(launch(std::integral_constant<int, 2>()));
    prev = !debug_sync();
    h->launches += 1;
  }
  return QBX_OK;
}
qbx_status launch_m2m_f32(qbx_handle* h, FmmPlan* f, cudaStream_t s) {
  return launch_fold<true>(h, f, s);
}
qbx_status launch_l2l_f32(qbx_handle* h, FmmPlan* f, cudaStream_t s) {
  return launch_fold<false>(h, f, s);
}

qbx_status launch_m2l_f32(qbx_handle* h, FmmPlan* f, cudaStream_t s) {
  if (f->n_vbox == 0 || f->n_m2l_items32 == 0) return QBX_OK;
  if (f->n_vsrc > 0) {
    mpole_to_f32_kernel<<<nblk(f->n_vsrc, kBoxGroup), kT, 0, s>>>(
        f->pb_max, f->m2l_vsrc.ptr, f->n_vsrc, f->box.level.ptr, f->lpb.ptr, f->eoff.ptr,
        f->conv.ptr, f->mpole.ptr, f->mu32.ptr);
    QBX_CUDA_TRY(cudaGetLastError());
    h->launches += 1;
  }
  int at = 0;
  auto gemm = [&](auto nt, int n) -> qbx_status {
    constexpr int NT = decltype(nt)::value;
    if (n > 0) {
      m2l_fold_kernel<NT><<<n, NT, 0, s>>>(
          f->m2l_items32.ptr + at, f->lpb.ptr, f->m2l_toff.ptr, f->m2l_frow.ptr, f->pb_max,
          f->m2l_rot.ptr, f->mu32.ptr, f->tm_f32.ptr, f->m2l_y.ptr);
      QBX_CUDA_TRY(cudaGetLastError());
      h->launches += 1;
    }
    at += n;
    return QBX_OK;
  };
  qbx_status st;
  if ((st = gemm(std::integral_constant<int, 128>(), f->n_m2l_width[0])) != QBX_OK) return st;
  if ((st = gemm(std::integral_constant<int, 96>(), f->n_m2l_width[1])) != QBX_OK) return st;
  if ((st = gemm(std::integral_constant<int, 64>(), f->n_m2l_width[2])) != QBX_OK) return st;
  m2l_f32_reduce_kernel<<<f->n_vbox, kT, 0, s>>>(
      f->pb_max, f->vbox.ptr, f->box.level.ptr, f->lpb.ptr, f->V.off.ptr, f->m2l_eyoff.ptr,
      f->m2l_y.ptr, f->conv.ptr, f->eoff.ptr, f->local.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  h->launches += 1;
  return QBX_OK;
}
