// Unevaluated sums of two float32 (high part x, low part y), about 45 bits of the value, for the step of
// the recursion over neighbouring m (zp_tri.h): rho (u + v) - d.  On the float32 pipe, which GB300 has 64
// times as much of as of float64.  (Two steps of a block in one packed instruction each: no faster.)
#pragma once

#include <cuda_runtime.h>

#include <cmath>

namespace zp {

// Each operation rounded by itself, no contraction (on the host: compiled with -ffp-contract=off).
#ifdef __CUDA_ARCH__
#define ZP_PAIR_OP(device, host) return device
#else
#define ZP_PAIR_OP(device, host) return host
#endif
__host__ __device__ __forceinline__ float pair_add(float a, float b) { ZP_PAIR_OP(__fadd_rn(a, b), a + b); }
__host__ __device__ __forceinline__ float pair_sub(float a, float b) { ZP_PAIR_OP(__fsub_rn(a, b), a - b); }
__host__ __device__ __forceinline__ float pair_mul(float a, float b) { ZP_PAIR_OP(__fmul_rn(a, b), a * b); }
__host__ __device__ __forceinline__ float pair_fma(float a, float b, float c) { ZP_PAIR_OP(__fmaf_rn(a, b, c), std::fmaf(a, b, c)); }
#undef ZP_PAIR_OP

// rho (u + v) - d: Knuth's exact sums of u + v and of the product minus d, the product's rounding by a
// fused operation, the low parts to first order.  The result is not renormalised: the high part runs
// the recursion in plain float32 (three operations from step to step) and the low part collects
// what its roundings leave out.
__host__ __device__ __forceinline__ float2 pair_step(float2 rho, float2 u, float2 v, float2 d) {
  const float s = pair_add(u.x, v.x), b = pair_sub(s, u.x);
  const float se = pair_add(pair_add(pair_sub(u.x, pair_sub(s, b)), pair_sub(v.x, b)), pair_add(u.y, v.y));
  const float p = pair_mul(rho.x, s);
  const float pe = pair_fma(rho.y, s, pair_fma(rho.x, se, pair_fma(rho.x, s, -p)));  // what p leaves out
  const float q = pair_sub(p, d.x), c = pair_sub(q, p);
  const float qe = pair_sub(pair_sub(p, pair_sub(q, c)), pair_add(d.x, c));
  return make_float2(q, pair_add(qe, pair_sub(pe, d.y)));
}

}  // namespace zp
