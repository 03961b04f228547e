// The float-float primitives of ff.cuh, one value (or one row) per thread, for
// test_ff_primitives_gpu.py. Inputs and outputs are host arrays.
#include "ff.cuh"

void set_error(const char*, ...) {}
cudaError_t dev_alloc(void** p, size_t n) { return cudaMalloc(p, n); }
void dev_free(void* p) { cudaFree(p); }

namespace {
__device__ ff get(double v) { return ff_round(v); }

__global__ void probe(int op, int n, const double* __restrict__ a, const double* __restrict__ b,
                      int iarg, FfUnits U, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (op == 0 || op == 1) {  // H_0, H_1 to 3 or 6 second parts
    ffh h0, h1;
    if (op == 0) hankel01_ff_any<3>(get(a[i]), h0, h1);
    else hankel01_ff_any<6>(get(a[i]), h0, h1);
    out[4 * i] = ff_f64(h0.x);
    out[4 * i + 1] = ff_f64(h0.y);
    out[4 * i + 2] = ff_f64(h1.x);
    out[4 * i + 3] = ff_f64(h1.y);
  } else if (op == 2) {  // v 2^-iarg
    out[i] = ff_f64(ff_from_f64(a[i], 896 + iarg));
  } else if (op == 3) {
    out[i] = ff_f64(ff_rsqrt(get(a[i])));
  } else if (op == 4) {  // 1 if not at the origin, k r, 1 / r (units of 2^-floor(log2 k)), direction
    FfPolar D;
    const bool off = D.set(a[i], b[i], U);
    double* o = out + 5 * i;
    o[0] = off;
    o[1] = off ? ff_f64(D.z) : 0.0;
    o[2] = off ? ff_f64(D.ir) : 0.0;
    o[3] = off ? D.c : 0.0;
    o[4] = off ? D.s : 0.0;
  } else if (op == 5) {  // FP32 back to FP64
    out[i] = f64_from_f32((float)a[i]);
  } else {  // J_0 .. J_M of |a|, M = op - 100, scaled by 2^{-iarg j}
    const int M = op - 100;
    float2 row[128];
    FfPolar D;
    D.set(a[i], 0.0, U);
    const ff inv = ff_miller_row(row, M, iarg, D, U);
    float sc = 1.f;
    for (int j = 0; j <= M; ++j) out[(size_t)i * (M + 1) + j] = ff_f64(ff_mul(ff_miller_value(row[j], sc), inv));
  }
}
}  // namespace

extern "C" int ff_probe(int op, int n, const double* a, const double* b, int iarg, double k,
                        int width, double* out) {
  if (n < 1 || op < 0 || (op > 5 && (op < 101 || op > 227))) return -1;
  double *da = nullptr, *db = nullptr, *dout = nullptr;
  cudaMalloc(&da, n * sizeof(double));
  cudaMalloc(&db, n * sizeof(double));
  cudaMalloc(&dout, (size_t)n * width * sizeof(double));
  cudaMemcpy(da, a, n * sizeof(double), cudaMemcpyHostToDevice);
  cudaMemcpy(db, b ? b : a, n * sizeof(double), cudaMemcpyHostToDevice);
  probe<<<(n + 63) / 64, 64>>>(op, n, da, db, iarg, make_ff_units(k), dout);
  cudaMemcpy(out, dout, (size_t)n * width * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(da);
  cudaFree(db);
  cudaFree(dout);
  return (int)cudaGetLastError();
}
