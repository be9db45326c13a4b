// Unevaluated sums of two float32 (high part x, low part y), about 45 bits of the value, for the step of the
// recursion over neighbouring m (zp_tri.h): rho (u + v) - d.  On the float32 pipe, which GB300 has 64
// times as much of as of float64; two independent steps share their instructions (f32x2).
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

namespace zp {

// Two float32 in one register pair, operated on by one instruction.
struct f32x2 {
  uint64_t v;
  __device__ __forceinline__ static f32x2 of(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
  }
  __device__ __forceinline__ void get(float& a, float& b) const { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
};
__device__ __forceinline__ f32x2 add_(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f32x2 sub_(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f32x2 mul_(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f32x2 fma_(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// Each operation rounded by itself, no contraction (on the host: compiled with -ffp-contract=off).
#ifdef __CUDA_ARCH__
#define ZP_PAIR_OP(device, host) return device
#else
#define ZP_PAIR_OP(device, host) return host
#endif
__host__ __device__ __forceinline__ float add_(float a, float b) { ZP_PAIR_OP(__fadd_rn(a, b), a + b); }
__host__ __device__ __forceinline__ float sub_(float a, float b) { ZP_PAIR_OP(__fsub_rn(a, b), a - b); }
__host__ __device__ __forceinline__ float mul_(float a, float b) { ZP_PAIR_OP(__fmul_rn(a, b), a * b); }
__host__ __device__ __forceinline__ float fma_(float a, float b, float c) { ZP_PAIR_OP(__fmaf_rn(a, b, c), std::fmaf(a, b, c)); }
#undef ZP_PAIR_OP

// rho = h + l as the step below reads it: h, -h and -l.
template <typename T>
struct PairFactor {
  T h, nh, nl;
};

// (h, l) = rho (u + v) - d: Knuth's exact sums of u + v and of the product minus d, the product's
// rounding by a fused operation, the low parts to first order.  The sum h + l is not renormalised:
// h runs the recursion in plain float32 (three operations from step to step) and l collects what its
// roundings leave out.
#pragma nv_exec_check_disable
template <typename T>
__host__ __device__ __forceinline__ void pair_core(const PairFactor<T>& r, T uh, T ul, T vh, T vl, T dh, T dl, T& h, T& l) {
  const T s = add_(uh, vh), b = sub_(s, uh);
  const T se = add_(add_(sub_(uh, sub_(s, b)), sub_(vh, b)), add_(ul, vl));
  const T p = mul_(r.h, s);
  const T ne = fma_(r.nl, s, fma_(r.nh, se, fma_(r.nh, s, p)));  // minus what p leaves out
  const T q = sub_(p, dh), c = sub_(q, p);
  h = q;
  l = sub_(sub_(sub_(p, sub_(q, c)), add_(dh, c)), add_(ne, dl));
}

__host__ __device__ __forceinline__ float2 pair_step(const PairFactor<float>& r, float2 u, float2 v, float2 d) {
  float2 e;
  pair_core<float>(r, u.x, u.y, v.x, v.y, d.x, d.y, e.x, e.y);
  return e;
}
__device__ __forceinline__ void pair_step2(const PairFactor<f32x2>& r, float2 u0, float2 v0, float2 d0, float2 u1, float2 v1, float2 d1,
                                           float2& e0, float2& e1) {
  f32x2 h, l;
  pair_core<f32x2>(r, f32x2::of(u0.x, u1.x), f32x2::of(u0.y, u1.y), f32x2::of(v0.x, v1.x), f32x2::of(v0.y, v1.y),
                   f32x2::of(d0.x, d1.x), f32x2::of(d0.y, d1.y), h, l);
  h.get(e0.x, e1.x);
  l.get(e0.y, e1.y);
}

}  // namespace zp
