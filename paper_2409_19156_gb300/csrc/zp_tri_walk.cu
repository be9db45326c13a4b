// Radial polynomials, rho-derivatives and Z over a whole triangle n <= n_max in float64, by the
// recursion over neighbouring m (see zp_tri.h for the layout and its derivation):
//   R_n^m = rho T_0 - R_{n-2}^m,   (R_n^m)^(k) = n T_{k-1} + (R_{n-2}^m)^(k),
//   T_k = (R_{n-1}^{|m-1|})^(k) + (R_{n-1}^{m+1})^(k)
// (the derivative form from U_n' = 2n U_{n-1} + U_{n-2}' under the integral).  A value costs 2, 3, 5
// or 7 float64 operations for k <= 0, 1, 2, 3 against the column recursion's 3, 7, 11 or 15 with its
// weights, needs no tables, and loses less: an error spreads with weights of at most 1 (radial set
// n <= 100, k = 0..3: 7e-16 of the norm against 6e-15), while values in the growth region near the
// origin add terms of one sign and keep their relative accuracy.
//
// One warp per 32 points, one point per thread, walking 2 x 2 blocks of (a, b) = ((n+m)/2, (n-m)/2)
// row by row; the row above (every lane of its derivatives) is kept in shared memory, private to the
// thread, so nothing synchronises.  Bound: float64 issue (a warp's operation holds its scheduler's
// pipe for 64 cycles); the stores are whole 128-byte lines per warp.  cos / sin(m theta) come from
// the fixed-point angle functions on the integer pipe, which is idle here.
//
// With the whole row in shared memory, high degrees leave room for one warp per scheduler, which
// keeps the pipe two thirds busy: the instructions between two float64 operations are not hidden.
// The wide form (radial, k >= 2) holds the row's two highest derivative lanes in tensor memory (each
// warp reads its own 32 lanes of it), so that two warps per scheduler fit: eight in a block that takes
// all of tensor memory, so one block per SM works at a time (where shared memory admits another, it waits
// for the first one's tensor memory).  Its float64 pipe is 90 % busy over whole waves.
//
// Measured against the column form: radial set n <= 100, k <= 3, 1e5 points 6.32 -> 3.66 ms (4.62
// with one warp per scheduler); Z and dZ/drho with dZ/dtheta, n <= 32, 99991 points 836 -> 631 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "zp_angles.cuh"
#include "zp_api_common.h"
#include "zp_internal.h"
#include "zp_ptx.cuh"
#include "zp_series_internal.h"
#include "zp_tri.h"

namespace zp {
namespace {

constexpr int W = 32;           // points per warp
constexpr int kWideWarps = 8;   // warps of a block that keeps part of its rows in tensor memory
constexpr int kWideLanes = 2;   // its value lanes there (the highest derivatives)
constexpr uint32_t kMaxBlockSmem = 232448 - 64, kSmemPerSm = 233472, kSmemPerBlock = 1024;
constexpr int kWideCols = 256;  // tensor memory columns per warp: two warps share a quadrant's 512

struct TriWalkArgs {
  const int32_t* perm;  // modes of every position (zp_tri.h), -1 for none
  const double* r;
  const double* theta;
  int64_t p_begin, p_end;  // points p_begin .. p_end - 1 of P
  int64_t P, J;
  double* out;
  double* out_dtheta;
  unsigned long long* rowmax;
  int n_max;
};

__host__ __device__ constexpr uint32_t walk_smem(int n_max, int kmax, bool ang) {
  return (uint32_t)(tri_state_rows(n_max) * (kmax + 1) * W * 8 + (n_max + 3) * 8 + (ang ? (n_max + 1) * W * 16 : 0));
}

constexpr uint32_t wide_smem(int n_max, int kmax) {
  return (uint32_t)(tri_state_rows(n_max) * (kmax + 1 - kWideLanes) * kWideWarps * W * 8 + (n_max + 3) * 8);
}
// Whether the wide form fits (tensor memory columns and shared memory of one block per SM) and the
// one-warp form leaves fewer than six warps per SM (1e5 points, wide against one-warp form: k <= 3, four
// per SM, n <= 100: 3.71 against 4.62 ms; five per SM, n <= 72, k <= 3: 2.02 against 2.14 ms, and n <= 100,
// k <= 2: 2.80 against 2.91 ms).
constexpr bool wide_fits(int n_max, int kmax, bool ang) {
  return !ang && kmax >= 2 && tri_state_rows(n_max) * kWideLanes * 2 <= kWideCols && wide_smem(n_max, kmax) <= kMaxBlockSmem &&
         walk_smem(n_max, kmax, false) + kSmemPerBlock > kSmemPerSm / 6;
}

// KMAX: highest rho-derivative; ANG: Z instead of R; DT (with ANG): also dZ/dtheta; WIDE: eight warps
// per block, the row's two highest derivative lanes in tensor memory.
template <int KMAX, bool ANG, bool DT, bool WIDE>
__global__ void __launch_bounds__(WIDE ? kWideWarps * W : W) tri_walk_kernel(TriWalkArgs a) {
  static_assert(!WIDE || (!ANG && KMAX >= 2));
  extern __shared__ double tri_smem[];
  __shared__ uint32_t tmem_base;
  constexpr int L = KMAX + 1, LS = WIDE ? L - kWideLanes : L;  // lanes; those in shared memory
  constexpr int kWarps = WIDE ? kWideWarps : 1;
  // Four blocks per iteration: no register moves between them (radial set n <= 100, k <= 3, 1e5 points
  // 4.12 -> 3.66 ms); Z was slower with it (0.63 -> 0.65 ms).
  constexpr int kUnroll = ANG ? 1 : 4;
  const int lane = threadIdx.x % W, warp = threadIdx.x / W, n_max = a.n_max, H = n_max / 2;
  double2* an = reinterpret_cast<double2*>(tri_smem) + lane;  // [m][lane]
  double* st = tri_smem + (ANG ? (size_t)(n_max + 1) * W * 2 : 0) + (size_t)warp * tri_state_rows(n_max) * LS * W + lane;  // [b][k][lane]
  double* num = tri_smem + (ANG ? (size_t)(n_max + 1) * W * 2 : 0) + (size_t)kWarps * tri_state_rows(n_max) * LS * W;  // 0, 1, 2, ..
  for (int i = threadIdx.x; i < n_max + 3; i += kWarps * W) num[i] = (double)i;
  uint32_t tm = 0;  // [b / 2][row of two][k][low, high word] of this thread's lane
  if constexpr (WIDE) {
    if (warp == 0) {
      ptx::tmem_alloc(&tmem_base, 2 * kWideCols);
      ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    tm = tmem_base + ((uint32_t)(warp % 4) << 21) + (uint32_t)(warp / 4) * kWideCols;
  } else {
    __syncwarp();
  }
  const int64_t p = a.p_begin + ((int64_t)blockIdx.x * kWarps + warp) * W + lane;
  const bool valid = p < a.p_end;
  const double rho = valid ? a.r[p] : 0.0;
  if constexpr (ANG)
    for_each_angle(valid ? a.theta[p] : 0.0, n_max, [&](int m, double c, double s) { an[(size_t)m * W] = make_double2(c, s); });
  double* const out = a.out + p;
  double* const out_dt = DT ? a.out_dtheta + p : nullptr;
  const int64_t order = a.J * a.P;

  auto put = [&](int32_t j, const double (&v)[L], double dt) {
    if (j < 0) return;
    double* o = out + (int64_t)j * a.P;
    if (valid) {
#pragma unroll
      for (int k = 0; k < L; ++k) __stcs(o + k * order, v[k]);
      if constexpr (DT) __stcs(out_dt + (int64_t)j * a.P, dt);
    }
    if constexpr (KMAX == 0 && ANG) {
      if (a.rowmax) {  // the row's largest high word, for the float64-accurate GEMM's scales
        const uint32_t h = valid ? (uint32_t)__double2hiint(v[0]) & 0x7fffffffu : 0u;
        const uint32_t mx = __reduce_max_sync(0xffffffffu, h);
        if (lane == 0) atomicMax(a.rowmax + j, (unsigned long long)mx << 32);
      }
    }
  };
  auto emit = [&](const double (&f)[L], int32_t jc, int32_t js, int m) {
    if constexpr (!ANG) {
      put(jc, f, 0.0);
      put(js, f, 0.0);
    } else {
      if (jc < 0 && js < 0) return;
      const double2 g = an[(size_t)m * W];
      double c[L], s[L];
#pragma unroll
      for (int k = 0; k < L; ++k) {
        c[k] = f[k] * g.x;
        s[k] = f[k] * g.y;
      }
      const double md = DT ? num[m] : 0.0;
      put(jc, c, DT ? -md * s[0] : 0.0);
      put(js, s, DT ? md * c[0] : 0.0);
    }
  };

  const int4* perm = reinterpret_cast<const int4*>(a.perm);
  int block = 0;
  for (int A = 0; A <= H; ++A) {
    const int nb = min(A, H - A);
    double l0[L], l1[L], dg[L];  // f(2A, 2B-1), f(2A+1, 2B-1), f(2A-1, 2B-1) and their derivatives
#pragma unroll
    for (int k = 0; k < L; ++k) l0[k] = l1[k] = dg[k] = 0.0;
    if (A == 0) dg[0] = -1.0;
#pragma unroll kUnroll
    for (int B = 0; B <= nb; ++B, ++block) {
      // The row above.  Its lanes in tensor memory arrive asynchronously: loaded for every block (also
      // those that do not use them, whose columns are the block's own) and waited for in the same
      // straight-line stretch, so that nothing can touch the registers in between.
      uint32_t v[8];
      if constexpr (WIDE) {
        __syncwarp();
        ptx::tmem_ld_32x32b_x8(tm + 8 * B, v);
      }
      const int4 jc = __ldg(perm + 2 * block), js = __ldg(perm + 2 * block + 1);
      double* row = st + (size_t)(2 * B) * LS * W;
      double u0[L], u1[L], e00[L], e01[L], e10[L], e11[L];
      if constexpr (WIDE) {
#pragma unroll
        for (int k = 0; k < LS; ++k) {
          u0[k] = row[k * W];
          u1[k] = row[(LS + k) * W];
        }
        ptx::tmem_ld_wait(v);
#pragma unroll
        for (int k = 0; k < kWideLanes; ++k) {
          u0[LS + k] = __hiloint2double((int)v[2 * k + 1], (int)v[2 * k]);
          u1[LS + k] = __hiloint2double((int)v[2 * k + 5], (int)v[2 * k + 4]);
        }
#pragma unroll
        for (int k = 0; k < L; ++k) {
          u0[k] = B < A ? u0[k] : l0[k];
          u1[k] = B < A ? u1[k] : l1[k];
        }
      } else {
#pragma unroll
        for (int k = 0; k < L; ++k) {
          u0[k] = B < A ? row[k * W] : l0[k];
          u1[k] = B < A ? row[(L + k) * W] : l1[k];
        }
      }
      const int n0 = 2 * (A + B), m0 = 2 * (A - B);
      const double nd0 = num[n0], nd1 = num[n0 + 1], nd2 = num[n0 + 2];
      // One element from its neighbours above and to the left and the one across.
      auto element = [&](double (&f)[L], const double (&up)[L], const double (&left)[L], const double (&old)[L], double n) {
        double t = up[0] + left[0];
        f[0] = fma(rho, t, -old[0]);
#pragma unroll
        for (int k = 1; k < L; ++k) {
          f[k] = fma(n, t, old[k]);
          if (k + 1 < L) t = up[k] + left[k];
        }
      };
      element(e00, u0, l0, dg, nd0);
      if (A == 0) e00[0] = 1.0;  // R_0^0, also of a radius that is not finite (0 rho would not be)
      element(e01, u1, e00, u0, nd1);
      element(e10, e00, l1, l0, nd1);
      element(e11, e01, e10, e00, nd2);
#pragma unroll
      for (int k = 0; k < L; ++k) {
        if (k < LS) {
          row[k * W] = e10[k];
          row[(LS + k) * W] = e11[k];
        }
        dg[k] = u1[k];
        l0[k] = e01[k];
        l1[k] = e11[k];
      }
      if constexpr (WIDE) {
        auto lo = [](double x) { return (uint32_t)__double2loint(x); };
        auto hi = [](double x) { return (uint32_t)__double2hiint(x); };
        ptx::tmem_st_32x32b_x4<0>(tm + 8 * B, lo(e10[LS]), hi(e10[LS]), lo(e10[LS + 1]), hi(e10[LS + 1]));
        ptx::tmem_st_32x32b_x4<4>(tm + 8 * B, lo(e11[LS]), hi(e11[LS]), lo(e11[LS + 1]), hi(e11[LS + 1]));
      }
      const TriAngleRows am = tri_angle_rows(m0, n_max);
      emit(e00, jc.x, js.x, am.mid);
      emit(e01, jc.y, js.y, am.low);
      emit(e10, jc.z, js.z, am.top);
      emit(e11, jc.w, js.w, am.mid);
    }
    if constexpr (WIDE) {  // before the next row's reads
      __syncwarp();
      ptx::tmem_st_wait();
    }
  }
  if constexpr (WIDE) {
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 0) ptx::tmem_dealloc(tmem_base, 2 * kWideCols);
  }
}

template <int KMAX, bool ANG, bool DT, bool WIDE>
cudaError_t launch(const TriWalkArgs& a, uint32_t smem, cudaStream_t st) {
  static DeviceMemo<int> memo;
  int set = 0;
  const zp_status s = memo.get(&set, [](int* x) -> zp_status {
    *x = 1;
    const cudaError_t e = cudaFuncSetAttribute(tri_walk_kernel<KMAX, ANG, DT, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)(WIDE ? kMaxBlockSmem : kTriWalkSmem));
    return e == cudaSuccess ? ZP_OK : cuda_error(e, "triangle walk set-up");
  });
  if (s != ZP_OK) return cudaErrorInvalidValue;
  constexpr int kPoints = WIDE ? kWideWarps * W : W;
  tri_walk_kernel<KMAX, ANG, DT, WIDE><<<(unsigned)((a.p_end - a.p_begin + kPoints - 1) / kPoints), kPoints, smem, st>>>(a);
  return cudaGetLastError();
}

template <int KMAX>
cudaError_t launch_k(TriWalkArgs a, int64_t wide, cudaStream_t st) {
  if constexpr (KMAX >= 2) {
    if (wide > 0) {
      TriWalkArgs b = a;
      b.p_end = wide;
      const cudaError_t e = launch<KMAX, false, false, true>(b, wide_smem(a.n_max, KMAX), st);
      if (e != cudaSuccess || wide == a.p_end) return e;
      a.p_begin = wide;
    }
  }
  const uint32_t smem = walk_smem(a.n_max, KMAX, a.theta != nullptr);
  if (a.theta == nullptr) return launch<KMAX, false, false, false>(a, smem, st);
  return a.out_dtheta ? launch<KMAX, true, true, false>(a, smem, st) : launch<KMAX, true, false, false>(a, smem, st);
}

}  // namespace

int64_t tri_walk_points(const zp_plan* plan, int64_t n_points, int max_deriv, bool ang, bool dtheta, int sms) {
  if (!plan->dev.tri_perm || walk_smem(plan->n_max, max_deriv, ang) > kTriWalkSmem) return 0;
  // Float64 operations per point of either form.
  const int64_t pairs = (int64_t)(plan->n_max / 2 + 1) * ((plan->n_max + 1) / 2 + 1);
  const int64_t per_value = max_deriv == 0 ? 2 : 2 * max_deriv + 1;
  const int64_t out_ops = ang ? plan->n_modes * (max_deriv + 1 + (dtheta ? 1 : 0)) : 0;
  int64_t steps = 0;
  for (const Column& c : plan->cols) steps += c.n_steps;
  const int64_t tri = pairs * per_value + out_ops, col = steps * (4 * max_deriv + 3) + out_ops;
  // The walk runs a warp per scheduler in whole waves of 4 sms warps; what is left over takes the
  // column form, which spreads a point over its columns.  An operation costs the walk about 4/3 of
  // the column form's time (its float64 pipe waits for shared memory and stores where the column
  // form's eight steps overlap: radial set n <= 100, k <= 3, one warp per scheduler: 440 against 622 G
  // operations/s).
  const int64_t wave = 4 * (int64_t)sms * W;
  int64_t points = n_points / wave * wave;
  const int64_t rest = n_points - points;
  if (3 * rest * col > 4 * wave * tri) points = n_points;
  return 4 * tri < 3 * col ? points : 0;
}

zp_status launch_tri_walk(const zp_plan* plan, const double* r, const double* theta, int64_t n_points, int64_t p_end,
                          int max_deriv, double* out, double* out_dtheta, unsigned long long* rowmax, int sms,
                          cudaStream_t stream) {
  TriWalkArgs a;
  a.perm = plan->dev.tri_perm;
  a.r = r;
  a.theta = theta;
  a.p_begin = 0;
  a.p_end = p_end;
  a.P = n_points;
  a.J = plan->n_modes;
  a.out = out;
  a.out_dtheta = out_dtheta;
  a.rowmax = rowmax;
  a.n_max = plan->n_max;
  const int64_t blocks = (p_end + W - 1) / W;
  if (blocks > 0x7fffffffLL) return set_error(ZP_ERR_INVALID_ARG, "n_points too large for one launch");
  // Whole waves of eight warps per SM in the wide form, what is left over one warp per scheduler.
  const int64_t wave = (int64_t)sms * kWideWarps * W;
  const int64_t wide = wide_fits(plan->n_max, max_deriv, theta != nullptr) ? p_end / wave * wave : 0;
  cudaError_t e;
  switch (max_deriv) {
    case 0: e = launch_k<0>(a, wide, stream); break;
    case 1: e = launch_k<1>(a, wide, stream); break;
    case 2: e = launch_k<2>(a, wide, stream); break;
    default: e = launch_k<3>(a, wide, stream); break;
  }
  return e == cudaSuccess ? ZP_OK : cuda_error(e, "tri_walk_kernel launch");
}

}  // namespace zp
