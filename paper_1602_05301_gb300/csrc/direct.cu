// All-pairs ("direct") kernels of Global QBX, FP64:
//   strengths      per-source charge / dipole strengths
//   p2qbxl_direct  QBX coefficients at every centre from every source
//                  (Sec. 7, Eq. (localexpcoeffs); double layer by the normal
//                  derivative of the Graf kernel)
//   p2p_direct     smooth Gauss quadrature at unassociated targets
//                  (Sec. 3.2, Eq. (gauss-layerpot))
//   qbxl2p         truncated J-expansion at associated targets (Sec. 2.1, Eq. (phiapprox))
//   associate      target association (Sec. 6.1) by exhaustive search
//   place_centres  c = s + side (h/2) n (Sec. 2.2)
#include <cmath>
#include <cstdio>

#include "qbx_internal.h"
#include "p2qbxl_pair.cuh"

namespace {

// q_j = (i/4) w_j cS sigmaS_j,  d_j = (i/4) w_j cD sigmaD_j; with str_exp each
// block's largest exponent
__global__ void __launch_bounds__(256) strengths_kernel(
    int64_t n, const double* __restrict__ w, cd cS, const cd* __restrict__ sS, cd cD,
    const cd* __restrict__ sD, cd* __restrict__ q, cd* __restrict__ d, int lk,
    int* __restrict__ str_exp) {
  int e = 0;
#pragma unroll 4
  for (int64_t j = blockIdx.x * (int64_t)256 + threadIdx.x; j < n; j += (int64_t)256 * gridDim.x) {
    const cd i4 = mk(0.0, 0.25 * w[j]);
    const cd qj = sS ? cmul(i4, cmul(cS, sS[j])) : mk(0.0, 0.0);
    const cd dj = sD ? cmul(i4, cmul(cD, sD[j])) : mk(0.0, 0.0);
    q[j] = qj;
    d[j] = dj;
    e = max(e, strength_exponent(qj, dj, lk));
  }
  if (!str_exp) return;
  e = block_exponent(e);
  if (threadIdx.x == 0) str_exp[blockIdx.x] = e;
}

// alpha at the centres list[0..n) (every centre when list is NULL), SW warps per
// centre and one centre per block: the lanes deal the sources round-robin, each
// keeps 2p+1 partial coefficients (p2qbxl_pair), a reduce-scatter of shuffles
// adds the lanes and, for SW > 1, the warps' sums are added in warp order
// through shared memory (deterministic). FP64-pipe-bound; what matters besides
// the instruction count is that every SM has a few warps: a thread per centre
// (the form before) put the 1024 centres of a circle on 8 of the 152 SMs.
// One-warp blocks even the load over the SMs to within one centre.
template <int PM, bool HS, bool HD, int SW>
__global__ void __launch_bounds__(32 * SW) p2qbxl_direct_kernel(
    const int32_t* __restrict__ list, const double* __restrict__ ctr_xy, int64_t n_src,
    const double* __restrict__ src_xy, const double* __restrict__ src_nrm,
    const cd* __restrict__ qs, const cd* __restrict__ ds, double k, int p,
    cd* __restrict__ alpha) {
  constexpr int NC = 2 * PM + 2;
  const int64_t c = list ? (int64_t)list[blockIdx.x] : (int64_t)blockIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const double cx = ctr_xy[2 * c], cy = ctr_xy[2 * c + 1];
  const double ik = 1.0 / k, hk = 0.5 * k;
  cd acc[NC];
#pragma unroll
  for (int i = 0; i < NC; ++i) acc[i] = mk(0.0, 0.0);
  for (int64_t j = threadIdx.x; j < n_src; j += 32 * SW) {
    const cd z = mk(0.0, 0.0);
    p2qbxl_pair<PM, HS, HD>(acc, src_xy[2 * j] - cx, src_xy[2 * j + 1] - cy, HS ? qs[j] : z,
                            HD ? cscale(ds[j], hk) : z, HD ? src_nrm[2 * j] : 0.0,
                            HD ? src_nrm[2 * j + 1] : 0.0, k, ik, p);
  }
  cd x32, x33;
  group_reduce_scatter<32, NC>(acc, lane, x32, x33);
  cd v = acc[0];
  if (SW > 1) {
    __shared__ cd part[SW][34];
    part[w][lane] = v;
    if (lane == 0) {
      part[w][32] = x32;
      part[w][33] = x33;
    }
    __syncthreads();
    if (w > 0) return;
    x32 = part[0][32];
    x33 = part[0][33];
    for (int u = 1; u < SW; ++u) {
      v = cadd(v, part[u][lane]);
      x32 = cadd(x32, part[u][32]);
      x33 = cadd(x33, part[u][33]);
    }
  }
  cd* dst = alpha + c * (2 * p + 1) + p;
  pair_coefficients<32, PM>(v, v, x32, x33, lane, p, [&](int l, cd a) { dst[l] = a; });
}

// Smooth quadrature: u(t) = sum_j q_j H_0(k r) + d_j k H_1(k r) n_j.(t - s_j)/r.
// A warp per target, the lanes over the sources, a shuffle tree; one-warp blocks
// for the same reason as above.
template <bool HS, bool HD>
__global__ void __launch_bounds__(32) p2p_direct_kernel(
    const int32_t* __restrict__ list, const double* __restrict__ tgt_xy, int64_t n_src,
    const double* __restrict__ src_xy, const double* __restrict__ src_nrm,
    const cd* __restrict__ qs, const cd* __restrict__ ds, double k, cd* __restrict__ out) {
  const int64_t t = list[blockIdx.x];
  const double tx = tgt_xy[2 * t], ty = tgt_xy[2 * t + 1], ik = 1.0 / k;
  cd acc = mk(0.0, 0.0);
  for (int64_t j = threadIdx.x; j < n_src; j += 32) {
    const double dx = tx - src_xy[2 * j], dy = ty - src_xy[2 * j + 1];
    const double r2 = dx * dx + dy * dy;
    if (r2 == 0.0) continue;
    const double ir = rsqrt(r2), x = k * (r2 * ir);
    cd h0, h1;
    hankel01_any<false, HS, HD>(x, ik * ir, h0, h1);
    if (HS) cfma(acc, qs[j], h0);
    if (HD) cfma(acc, ds[j], cscale(h1, k * (src_nrm[2 * j] * dx + src_nrm[2 * j + 1] * dy) * ir));
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
    acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
  }
  if (threadIdx.x == 0) out[t] = acc;
}

// u(t) = sum_{|l| <= p} alpha_l(c) J_l(k rho) e^{-i l theta}, (rho, theta) the
// polar coordinates of t - c (Eq. (phiapprox)); J_{-m} = (-1)^m J_m.
template <int PM>
__device__ __forceinline__ cd qbx_local_eval(double tx, double ty, const double* __restrict__ ctr_xy,
                                             int64_t c, const cd* __restrict__ alpha, double k,
                                             int p) {
  const double dx = tx - ctr_xy[2 * c];
  const double dy = ty - ctr_xy[2 * c + 1];
  const double rho = sqrt(dx * dx + dy * dy);
  const cd e1 = rho > 0.0 ? mk(dx / rho, dy / rho) : mk(1.0, 0.0);
  double J[PM + 1];
  bessel_j_array<PM>(k * rho, J);
  const int P = 2 * p + 1;
  const cd* a = alpha + c * P + p;  // a[l], l = -p..p
  cd u = cscale(a[0], J[0]);
  cd e = mk(1.0, 0.0);
  double sgn = 1.0;
#pragma unroll
  for (int m = 1; m <= PM; ++m) {
    if (m > p) break;
    e = cmul(e, e1);
    sgn = -sgn;
    cfma(u, cscale(a[m], J[m]), cconj(e));
    cfma(u, cscale(a[-m], sgn * J[m]), e);
  }
  return u;
}

// QBX evaluation at the associated targets. A target marked in avg (an
// on-surface target asking for the on-surface value) gets the mean of its
// node's exterior (assoc) and interior (assoc + n_nodes) one-sided limits
// (Sec. 2, Eq. (oneside): the two limits differ by the jump of D).
template <int PM>
__global__ void __launch_bounds__(128) qbxl2p_kernel(int64_t n_list, const int32_t* __restrict__ list,
                                                     const double* __restrict__ tgt_xy,
                                                     const int32_t* __restrict__ assoc,
                                                     const int8_t* __restrict__ avg,
                                                     int64_t n_nodes,
                                                     const double* __restrict__ ctr_xy,
                                                     const cd* __restrict__ alpha, double k,
                                                     int p, cd* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n_list) return;
  const int64_t t = list[i];
  const int64_t c = assoc[t];
  const double tx = tgt_xy[2 * t], ty = tgt_xy[2 * t + 1];
  cd u = qbx_local_eval<PM>(tx, ty, ctr_xy, c, alpha, k, p);
  if (avg && avg[t]) {
    const cd v = qbx_local_eval<PM>(tx, ty, ctr_xy, c + n_nodes, alpha, k, p);
    u = mk(0.5 * (u.x + v.x), 0.5 * (u.y + v.y));
  }
  out[t] = u;
}

// Exhaustive association, arithmetic without contraction so that ties and
// boundaries are decided exactly as in a plain IEEE evaluation.
__global__ void associate_direct_kernel(int64_t n_tgt, const double* __restrict__ tgt_xy,
                                        const int64_t* __restrict__ on_node,
                                        const int8_t* __restrict__ on_side, int64_t n_nodes,
                                        const double* __restrict__ node_xy,
                                        const double* __restrict__ panel_h, int q,
                                        int64_t n_ctr, const double* __restrict__ ctr_xy,
                                        const double* __restrict__ ctr_r, double eps,
                                        int32_t* __restrict__ assoc, int32_t* __restrict__ ctrs) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n_tgt) return;
  if (on_node && on_node[t] >= 0) {
    const int64_t j = on_node[t];
    const int side = on_side ? on_side[t] : 1;
    assoc[t] = (int32_t)(side >= 0 ? j : n_nodes + j);
    return;
  }
  const double tx = tgt_xy[2 * t], ty = tgt_xy[2 * t + 1];
  const double one_eps = __dadd_rn(1.0, eps);
  int64_t best = -1;
  double best_d2 = 1.0 / 0.0;
  for (int64_t c = 0; c < n_ctr; ++c) {
    const double dx = __dsub_rn(tx, ctr_xy[2 * c]);
    const double dy = __dsub_rn(ty, ctr_xy[2 * c + 1]);
    const double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
    const double lim = __dmul_rn(one_eps, ctr_r[c]);
    if (d2 <= __dmul_rn(lim, lim) && d2 < best_d2) {
      best = c;
      best_d2 = d2;
    }
  }
  if (best >= 0) {
    assoc[t] = (int32_t)best;
    return;
  }
  for (int64_t j = 0; j < n_nodes; ++j) {
    const double dx = __dsub_rn(tx, node_xy[2 * j]);
    const double dy = __dsub_rn(ty, node_xy[2 * j + 1]);
    const double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
    const double qh = __dmul_rn(0.25, panel_h[j / q]);
    if (d2 <= __dmul_rn(qh, qh)) {
      assoc[t] = -2;
      atomicAdd(&ctrs[0], 1);
      atomicMin(&ctrs[1], (int32_t)t);
      return;
    }
  }
  assoc[t] = -1;
}

__global__ void place_centres_kernel(int64_t n, int q, int sides, const double* __restrict__ node_xy,
                                     const double* __restrict__ node_nrm,
                                     const double* __restrict__ panel_h,
                                     double* __restrict__ ctr_xy, double* __restrict__ ctr_r) {
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= n) return;
  const double h = panel_h[j / q];
  for (int s = 0; s < sides; ++s) {
    const double a = (s == 0 ? 0.5 : -0.5) * h;  // exact: power-of-two scaling
    const int64_t c = j + s * n;
    ctr_xy[2 * c] = __dadd_rn(node_xy[2 * j], __dmul_rn(a, node_nrm[2 * j]));
    ctr_xy[2 * c + 1] = __dadd_rn(node_xy[2 * j + 1], __dmul_rn(a, node_nrm[2 * j + 1]));
    ctr_r[c] = 0.5 * h;
  }
}

inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// Warps per centre: one while the centres alone give every SM kWarpsPerSm warps
// (enough to keep the FP64 pipe busy), else four, as long as that leaves every
// lane a source.
constexpr int64_t kWarpsPerSm = 6;

template <int PM, bool HS, bool HD>
void p2qbxl_direct_launch(int64_t n, const int32_t* list, const double* cxy, int64_t n_src,
                          const double* sxy, const double* snrm, const cd* q, const cd* d,
                          double k, int p, cd* alpha, cudaStream_t s) {
  if (n >= 152 * kWarpsPerSm || n_src < 128)
    p2qbxl_direct_kernel<PM, HS, HD, 1><<<(unsigned)n, 32, 0, s>>>(list, cxy, n_src, sxy, snrm, q,
                                                                   d, k, p, alpha);
  else
    p2qbxl_direct_kernel<PM, HS, HD, 4><<<(unsigned)n, 128, 0, s>>>(list, cxy, n_src, sxy, snrm, q,
                                                                    d, k, p, alpha);
}

// alpha at n centres (list, or 0..n-1 when it is NULL) from every source
template <int PM>
void p2qbxl_direct_flags(int64_t n, const int32_t* list, const double* cxy, int64_t n_src,
                         const double* sxy, const double* snrm, const cd* q, const cd* d, bool S,
                         bool D, double k, int p, cd* alpha, cudaStream_t s) {
  if (S && D)
    p2qbxl_direct_launch<PM, true, true>(n, list, cxy, n_src, sxy, snrm, q, d, k, p, alpha, s);
  else if (S)
    p2qbxl_direct_launch<PM, true, false>(n, list, cxy, n_src, sxy, snrm, q, d, k, p, alpha, s);
  else
    p2qbxl_direct_launch<PM, false, true>(n, list, cxy, n_src, sxy, snrm, q, d, k, p, alpha, s);
}

void p2qbxl_direct(int64_t n, const int32_t* list, const double* cxy, int64_t n_src,
                   const double* sxy, const double* snrm, const cd* q, const cd* d, bool S, bool D,
                   double k, int p, cd* alpha, cudaStream_t s) {
  if (p <= 4) p2qbxl_direct_flags<4>(n, list, cxy, n_src, sxy, snrm, q, d, S, D, k, p, alpha, s);
  else if (p <= 8) p2qbxl_direct_flags<8>(n, list, cxy, n_src, sxy, snrm, q, d, S, D, k, p, alpha, s);
  else if (p <= 12) p2qbxl_direct_flags<12>(n, list, cxy, n_src, sxy, snrm, q, d, S, D, k, p, alpha, s);
  else p2qbxl_direct_flags<16>(n, list, cxy, n_src, sxy, snrm, q, d, S, D, k, p, alpha, s);
}

}  // namespace

qbx_status launch_strengths(qbx_handle* h, cd cS, const cd* sigS, cd cD, const cd* sigD,
                            cudaStream_t s) {
  if (h->n_src == 0) return QBX_OK;
  strengths_kernel<<<strength_blocks(h->n_src), 256, 0, s>>>(
      h->n_src, h->src_w.ptr, cS, sigS, cD, sigD, h->q_str.ptr, h->d_str.ptr, std::ilogb(h->k),
      h->str_exp.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  h->launches += 1;
  return QBX_OK;
}

qbx_status launch_p2qbxl_direct(qbx_handle* h, bool S, bool D, bool all_centres, cudaStream_t s) {
  if (h->n_ctr == 0) return QBX_OK;
  if (!S && !D) {
    QBX_CUDA_TRY(cudaMemsetAsync(h->alpha.ptr, 0, h->alpha.n * sizeof(cd), s));
    return QBX_OK;
  }
  // every centre when the caller reads the coefficients, else those that some
  // target is associated with (the only ones QBXL2P reads), as in FMM mode
  const int64_t n = all_centres ? h->n_ctr : h->n_used_ctr;
  if (n == 0) return QBX_OK;
  p2qbxl_direct(n, all_centres ? nullptr : h->used_ctr.ptr, h->ctr_xy.ptr, h->n_src,
                h->src_xy.ptr, h->src_nrm.ptr, h->q_str.ptr, h->d_str.ptr, S, D, h->k, h->p,
                h->alpha.ptr, s);
  QBX_CUDA_TRY(cudaGetLastError());
  h->launches += 1;
  return QBX_OK;
}

qbx_status launch_p2p_direct(qbx_handle* h, bool S, bool D, cd* out, cudaStream_t s) {
  const int64_t n = h->n_direct_tgt;
  if (n == 0) return QBX_OK;
#define P2P_DIRECT_LAUNCH(HS, HD)                                                              \
  p2p_direct_kernel<HS, HD><<<(unsigned)n, 32, 0, s>>>(                                        \
      h->direct_tgt_list.ptr, h->tgt_xy.ptr, h->n_src, h->src_xy.ptr, h->src_nrm.ptr,          \
      h->q_str.ptr, h->d_str.ptr, h->k, out)
  if (S && D) P2P_DIRECT_LAUNCH(true, true);
  else if (S) P2P_DIRECT_LAUNCH(true, false);
  else if (D) P2P_DIRECT_LAUNCH(false, true);
  else P2P_DIRECT_LAUNCH(false, false);
#undef P2P_DIRECT_LAUNCH
  QBX_CUDA_TRY(cudaGetLastError());
  h->launches += 1;
  return QBX_OK;
}

qbx_status launch_qbxl2p(qbx_handle* h, cd* out, cudaStream_t s) {
  const int64_t n = h->n_qbx_tgt;
  if (n == 0) return QBX_OK;
  dim3 g(nblk(n, 128));
  const int8_t* avg = h->has_avg ? h->avg.ptr : nullptr;
#define QBXL2P_LAUNCH(PM)                                                                  \
  qbxl2p_kernel<PM><<<g, 128, 0, s>>>(n, h->qbx_tgt_list.ptr, h->tgt_xy.ptr, h->assoc.ptr, \
                                      avg, h->n_nodes, h->ctr_xy.ptr, h->alpha.ptr, h->k,  \
                                      h->p, out)
  if (h->p <= 4) QBXL2P_LAUNCH(4);
  else if (h->p <= 8) QBXL2P_LAUNCH(8);
  else if (h->p <= 12) QBXL2P_LAUNCH(12);
  else QBXL2P_LAUNCH(16);
#undef QBXL2P_LAUNCH
  QBX_CUDA_TRY(cudaGetLastError());
  h->launches += 1;
  return QBX_OK;
}

qbx_status launch_associate_direct(qbx_handle* h, const int64_t* on_node, const int8_t* on_side,
                                   double eps, cudaStream_t s) {
  if (h->n_tgt == 0) return QBX_OK;
  associate_direct_kernel<<<nblk(h->n_tgt, 128), 128, 0, s>>>(
      h->n_tgt, h->tgt_xy.ptr, on_node, on_side, h->n_nodes, h->node_xy.ptr, h->panel_h.ptr,
      h->q, h->n_ctr, h->ctr_xy.ptr, h->ctr_r.ptr, eps, h->assoc.ptr, h->counters.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  return QBX_OK;
}

qbx_status launch_place_centres(qbx_handle* h, cudaStream_t s) {
  if (h->n_nodes == 0) return QBX_OK;
  place_centres_kernel<<<nblk(h->n_nodes, 256), 256, 0, s>>>(
      h->n_nodes, h->q, h->sides, h->node_xy.ptr, h->node_nrm.ptr, h->panel_h.ptr, h->ctr_xy.ptr,
      h->ctr_r.ptr);
  QBX_CUDA_TRY(cudaGetLastError());
  return QBX_OK;
}

// ---------------------------------------------------------------- allocation-free entry point
// qbx_direct_qbx_eval_noalloc: the direct QBX evaluation (strengths -> coefficients
// at every centre from every source -> J-expansion at each target) for callers
// that may not allocate device memory. Its scratch (strengths and coefficients)
// is the file-scope array below, reserved once per device when the library's
// module loads and shared by every call on that device.
#include <mutex>

namespace {

constexpr int64_t kNoAllocScratch = int64_t(1) << 19;  // complex doubles = 8 MiB per device
static __device__ __align__(256) cd g_noalloc_scratch[kNoAllocScratch];

constexpr int kNoAllocMaxDevices = 128;
std::mutex g_noalloc_mu;
cd* g_noalloc_ptr[kNoAllocMaxDevices] = {};

// J-expansion of centre centre[t] at target t (Eq. (phiapprox)); an out-of-range
// centre index yields NaN for that target.
template <int PM>
__global__ void __launch_bounds__(128) qbxl2p_each_kernel(int64_t n_tgt,
                                                          const double* __restrict__ tgt_xy,
                                                          const int32_t* __restrict__ centre,
                                                          int64_t n_ctr,
                                                          const double* __restrict__ ctr_xy,
                                                          const cd* __restrict__ alpha, double k,
                                                          int p, cd* __restrict__ out) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n_tgt) return;
  const int64_t c = centre[t];
  if (c < 0 || c >= n_ctr) {
    out[t] = mk(__longlong_as_double(0x7ff8000000000000LL), __longlong_as_double(0x7ff8000000000000LL));
    return;
  }
  const double dx = tgt_xy[2 * t] - ctr_xy[2 * c];
  const double dy = tgt_xy[2 * t + 1] - ctr_xy[2 * c + 1];
  const double rho = sqrt(dx * dx + dy * dy);
  const cd e1 = rho > 0.0 ? mk(dx / rho, dy / rho) : mk(1.0, 0.0);
  double J[PM + 1];
  bessel_j_array<PM>(k * rho, J);
  const int P = 2 * p + 1;
  const cd* a = alpha + c * P + p;
  cd u = cscale(a[0], J[0]);
  cd e = mk(1.0, 0.0);
  double sgn = 1.0;
#pragma unroll
  for (int m = 1; m <= PM; ++m) {
    if (m > p) break;
    e = cmul(e, e1);
    sgn = -sgn;
    cfma(u, cscale(a[m], J[m]), cconj(e));
    cfma(u, cscale(a[-m], sgn * J[m]), e);
  }
  out[t] = u;
}

// True if p is device (or managed) memory that belongs to device `dev`: a
// pointer into another GPU's memory would be dereferenced through peer access
// (or fault without it), so it is rejected like host memory.
bool on_device(const void* p, int dev) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) && a.device == dev;
}

}  // namespace

extern "C" qbx_status qbx_direct_qbx_eval_noalloc(
    int64_t n_src, const double* src_xy, const double* src_normal_xy, const double* src_weight,
    double k, double cS_re, double cS_im, const double* sigma_S, double cD_re, double cD_im,
    const double* sigma_D, int64_t n_ctr, const double* ctr_xy, int32_t p, int64_t n_tgt,
    const double* tgt_xy, const int32_t* tgt_centre, double* out, void* cuda_stream) {
  set_error("%s", "");
  if (n_src < 0 || n_ctr < 0 || n_tgt < 0 || p < 0 || p > QBX_MAX_P || !(k > 0.0)) {
    set_error("qbx_direct_qbx_eval_noalloc: invalid size, order or wavenumber");
    return QBX_ERR_ARG;
  }
  if (!sigma_S && !sigma_D) {
    set_error("qbx_direct_qbx_eval_noalloc: at least one of sigma_S, sigma_D is required");
    return QBX_ERR_ARG;
  }
  const int64_t P = 2 * (int64_t)p + 1;
  // 2 n_src + n_ctr P <= kNoAllocScratch, checked term by term so that no
  // product can overflow
  if (n_src > kNoAllocScratch / 2 || n_ctr > (kNoAllocScratch - 2 * n_src) / P) {
    set_error("qbx_direct_qbx_eval_noalloc: n_src = %lld and n_ctr = %lld at p = %d need "
              "2*n_src + n_ctr*(2p+1) complex scratch values but the static scratch holds %lld",
              (long long)n_src, (long long)n_ctr, p, (long long)kNoAllocScratch);
    return QBX_ERR_ARG;
  }
  int dev = 0;
  QBX_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kNoAllocMaxDevices) {
    set_error("qbx_direct_qbx_eval_noalloc: device ordinal %d not supported", dev);
    return QBX_ERR_ARG;
  }
  static const char* const names[] = {"src_xy", "src_normal_xy", "src_weight", "ctr_xy",
                                      "tgt_xy", "tgt_centre", "out", "sigma_S", "sigma_D"};
  const void* dev_ptrs[] = {src_xy, src_normal_xy, src_weight, ctr_xy, tgt_xy,
                            tgt_centre, out, sigma_S, sigma_D};
  const int64_t sizes[] = {n_src, n_src, n_src, n_ctr, n_tgt, n_tgt, n_tgt,
                           sigma_S ? n_src : 0, sigma_D ? n_src : 0};
  for (int i = 0; i < 9; ++i)
    if (sizes[i] > 0 && (!dev_ptrs[i] || !on_device(dev_ptrs[i], dev))) {
      set_error("qbx_direct_qbx_eval_noalloc: %s must be device memory on the current "
                "device (%d)", names[i], dev);
      return QBX_ERR_ARG;
    }
  cd* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      void* ptr = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
      if (e != cudaSuccess || !ptr) {
        set_error("qbx_direct_qbx_eval_noalloc: cudaGetSymbolAddress failed: %s",
                  cudaGetErrorString(e));
        return QBX_ERR_CUDA;
      }
      g_noalloc_ptr[dev] = (cd*)ptr;
    }
    scratch = g_noalloc_ptr[dev];
  }
  if (n_src == 0 && n_tgt == 0) return QBX_OK;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  cd* q = scratch;
  cd* d = scratch + n_src;
  cd* alpha = scratch + 2 * n_src;
  if (n_src > 0)
    strengths_kernel<<<nblk(n_src, 256), 256, 0, s>>>(
        n_src, src_weight, mk(cS_re, cS_im), (const cd*)sigma_S, mk(cD_re, cD_im),
        (const cd*)sigma_D, q, d, 0, nullptr);
  if (n_ctr > 0)
    p2qbxl_direct(n_ctr, nullptr, ctr_xy, n_src, src_xy, src_normal_xy, q, d, sigma_S != nullptr,
                  sigma_D != nullptr, k, p, alpha, s);
  if (n_tgt > 0) {
    const unsigned g = nblk(n_tgt, 128);
    cd* o = (cd*)out;
    if (p <= 4)
      qbxl2p_each_kernel<4><<<g, 128, 0, s>>>(n_tgt, tgt_xy, tgt_centre, n_ctr, ctr_xy, alpha, k, p, o);
    else if (p <= 8)
      qbxl2p_each_kernel<8><<<g, 128, 0, s>>>(n_tgt, tgt_xy, tgt_centre, n_ctr, ctr_xy, alpha, k, p, o);
    else if (p <= 12)
      qbxl2p_each_kernel<12><<<g, 128, 0, s>>>(n_tgt, tgt_xy, tgt_centre, n_ctr, ctr_xy, alpha, k, p, o);
    else
      qbxl2p_each_kernel<16><<<g, 128, 0, s>>>(n_tgt, tgt_xy, tgt_centre, n_ctr, ctr_xy, alpha, k, p, o);
  }
  QBX_CUDA_TRY(cudaGetLastError());
  return QBX_OK;
}
