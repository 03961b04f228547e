#pragma once

// Packed pairs of FP32 values (fma.rn.f32x2 and its kin, sm_100 and later): one
// issue slot for two FMAs, each rounded as the scalar instruction rounds it. The
// tile GEMMs were bound by issue (64 % of the slots, the FMA pipe at 53 %): M2L of
// 200 ellipses 4.03 -> 3.37 ms, M2M 0.83 -> 0.70 ms.
typedef unsigned long long f32p;
__device__ __forceinline__ f32p pk(float a, float b) {
  f32p r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpk(f32p v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32p fma2(f32p a, f32p b, f32p c) {
  f32p r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32p mul2(f32p a, f32p b) {
  f32p r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32p add2(f32p a, f32p b) {
  f32p r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32p sub2(f32p a, f32p b) { return fma2(b, pk(-1.f, -1.f), a); }

// s += y, where y holds the lost part n of the sum so far (s + n is the sum); the new
// lost part
__device__ __forceinline__ void kahan_add2(f32p& s, f32p& n, f32p y) {
  const f32p t = add2(s, y);
  n = sub2(y, sub2(t, s));
  s = t;
}
