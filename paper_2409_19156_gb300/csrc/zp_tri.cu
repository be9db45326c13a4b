// Fused float64-accurate Zernike series for up to 16 coefficient sets, every function of the
// triangle n <= n_max evaluated in fixed point on the integer pipe (zp_tri.h) and fed as digits
// through tensor memory to the tensor cores; no basis value, digit or partial sum goes to
// global memory.
//
//   values:     F[p, s]    = sum_j Z_j(p) C[j, s]
//   gradients:  grad_r[p]  = sum_s G[p, s] dF/dr,    grad_theta[p] = sum_s G[p, s] dF/dtheta
//
// The contraction is error-free slicing as in zp_fused.cu (digits of values and coefficients,
// diagonal sums exact in float32, recombined in integers), with 9 digits of 6 bits: values carry
// 53 fraction bits after |y| <= 1, coefficients 54 below their set's power-of-two scale.
//
// Gradients use that the derivatives of Zernike functions are sums of Zernike functions of lower
// degree: with V_n^m = R_n^m e^{i m theta} (m may be negative),
//   (d/dx -+ i d/dy) V_n^m = sum_{k = n, n-2, ..} 2 k V_{k-1}^{m -+ 1},
// so dF/dx and dF/dy are two more series over the same triangle, with coefficients formed once
// per call (tri_deriv_kernel), and one pass over the points contracts both:
//   dF/dr = cos F_x + sin F_y,   dF/dtheta = r (cos F_y - sin F_x).
//
// One persistent CTA per SM works through 128-point tiles, TMEM lane and point row alike:
//  - warps 8-11 (one per quadrant of 32 points) walk the triangle's 2 x 2 blocks from one stored
//    row in shared memory and hand the radial values on through a ring, two blocks per slot;
//  - warps 0-7 (two per quadrant, taking the chunks in turn) multiply them by the angle table
//    that they build per tile, cut the products into 9 digits (float16, exact) and store those as
//    the A operand in tensor memory (tcgen05.st: the digits never touch shared memory, whose
//    bandwidth the operand reads would share);
//  - warp 12 issues the MMAs: per chunk of 16 positions and digit one tcgen05.mma of N = 144 (9
//    diagonal blocks of 16 sets) against the coefficient digits shifted by that digit's blocks
//    (zero blocks in front), for each of the launch's coefficient groups;
//  - warp 13 copies the chunks' coefficient digits into shared memory (bulk copies);
//  - warps 0-7 drain finished accumulators.  One group: two accumulators, the previous segment
//    drained after the next is produced.  Two groups (gradients): both accumulators hold one
//    tile, drained before the next tile's first chunk.
// Points off the unit disc (or at angles of 2^52 and more) make their quadrant take the same walk in
// float64, with a row scale of its own per point: a walk more, and three to four times the time.  A
// 1000 x 1000 pixel grid over the square, n <= 32, 16 sets: 4.5 ms for values and 6.0 for gradients (the column
// form 10.4 and 25.4); the same points in random order, where every quadrant has one off the disc, 8.1
// and 8.3 (23.6 and 58.2).
//
// Bound: the integer instructions of the digit warps and their latencies (issue slots 56 %, ALU pipe
// 55 %, tensor pipe 31 % busy).  1e6 points r = sqrt(U), 561 modes, 16 sets: 2.30 ms, against 3.91 ms
// of the float64 column walk in zp_fused.cu, with a quarter of its error; both point gradients of
// 300007 such points in one pass instead of two.  Measured on the way there: eight warps that each
// walk and cut, one cos and one sin warp per quadrant 3.3 ms, with the multiplications in unsigned
// carries 2.7, in straight-line chunks 2.6; the walk in warps of its own 3.4, with eight stages of
// coefficient digits ahead instead of three 2.4.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "zp_api_common.h"
#include "zp_emu_device.cuh"
#include "zp_fused.h"
#include "zp_ptx.cuh"
#include "zp_series_internal.h"
#include "zp_tri.h"
#include "zp_tri_host.h"

namespace zp {
namespace {

constexpr int TM = 128;                      // points per tile (TMEM lanes)
constexpr int TND = kTriDigits;
constexpr int TNS = kFusedMaxSets;           // sets per diagonal block
constexpr int kDigitWarps = 8;               // warps 0-7: quadrant w % 4, group w / 4
constexpr int kWalkWarp = kDigitWarps;       // warps 8-11
constexpr int kMmaWarp = kWalkWarp + 4;      // and the copy warp after it
constexpr int kThreads = 32 * (kMmaWarp + 2);
constexpr int kRing = 4;                     // slots of radial values, a chunk each
constexpr uint32_t kRowB = 32;               // bytes of a coefficient row: one K step of 16 float16
constexpr uint32_t kBlockB = TNS * kRowB;    // one digit's block: 512 bytes
constexpr uint32_t kZeroB = (TND - 1) * kBlockB;
constexpr int kAccCols = TND * TNS;          // 144
constexpr int kStages = 3;                   // chunks of digits in tensor memory
constexpr int kMaxBStages = 8;               // chunks of coefficient digits in shared memory
constexpr int kAStage = TND * 8;             // TMEM columns of a chunk's digits
constexpr int kABase = 2 * kAccCols;
constexpr int kTmemCols = 512;
static_assert(kABase + kStages * kAStage <= kTmemCols, "tensor memory");
static_assert(kTriGroupBytes == TND * kBlockB, "coefficient digits of a chunk");
constexpr uint32_t kAux = 768;              // barriers and constants
constexpr uint32_t kSwapB = 2 * TM * 8;     // gradients: a point's two half sums
constexpr uint32_t kSlotB = 8 * TM * 8;     // a ring slot's values
constexpr uint32_t kRingB = kRing * (kSlotB + TM * 4);  // and its rows' scales
constexpr uint32_t kMaxSmem = 232448;
constexpr int kRowScale = 62;                // a value of row scale E is digitised at 2^(62 - E); E = 1 on the disc

// Bytes of a stage's coefficient operand.  One group: 8 zero blocks, then its digits.  Two: the
// second group's digits in reverse order, 8 zero blocks, the first group's digits, so that both
// share the zero blocks (the second group's accumulator then holds its diagonals in reverse).
__host__ __device__ constexpr uint32_t stage_bytes(int groups) { return kZeroB + (uint32_t)groups * kTriGroupBytes; }
__host__ __device__ constexpr uint32_t state_bytes(int n_max) { return (uint32_t)tri_state_rows(n_max) * TM * 8u; }
__host__ __device__ constexpr uint32_t angle_bytes(int n_max) { return (uint32_t)(n_max + 1) * TM * 16u; }
__host__ __device__ constexpr uint32_t smem_bytes(int n_max, int groups, int stages) {
  return 256u + kAux + (groups == 2 ? kSwapB : 0u) + kRingB + state_bytes(n_max) + angle_bytes(n_max) +
         (uint32_t)stages * stage_bytes(groups);
}
static_assert(smem_bytes(kTriMaxN, 2, 2) <= kMaxSmem, "two stages at the largest degree");

__device__ unsigned int g_tri_error = 0;  // set when a bounded wait gives up

// Constants of the digit cut, read from shared memory into registers: an instruction takes one
// immediate, so as constants known to the compiler each mask-and-merge is two instructions.
struct DigitConst {
  uint32_t pattern;             // 1024 twice
  uint32_t mask7, mask6, mask6_2, mask6_4;  // fields of 7 bits at 0, of 6 bits at 0, 2 and 4
  uint32_t minus7, minus6, minus6_2, minus6_4, scale_2, scale_4;
};
struct Barriers {
  uint64_t full[kStages];       // the four digit warps of a chunk's group
  uint64_t empty[kStages];      // MMA commit
  uint64_t bfull[kMaxBStages];  // coefficient copy
  uint64_t bempty[kMaxBStages];  // MMA commit
  uint64_t tfull[2];           // MMA commit after a segment's last chunk
  uint64_t tempty[2];          // digit warps after draining
  uint64_t rfull[kRing][4], rempty[kRing][4];  // ring slots, per quadrant
  uint64_t table_ready[4], table_free[4];      // angle table, per quadrant: its two digit warps
  uint64_t swap_full[4], swap_empty[4];  // gradients: a point's two halves (per quadrant)
  uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
  DigitConst digits;
};
static_assert(sizeof(Barriers) <= kAux, "barrier block");

__device__ __forceinline__ void fail(volatile int* abort_flag) {
  *abort_flag = 1;
  atomicOr(&g_tri_error, 1u);
}

__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int lane) {
  bool ok = true;
  if (lane == 0) ok = ptx::mbar_wait(bar, parity, abort_flag);
  return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
}

__device__ __forceinline__ const TriInst& inst_of(const TriArgs& a, int i) { return a.insts ? a.insts[i] : a.single; }
__device__ __forceinline__ void item_of(const TriArgs& a, int64_t it, int& inst, int64_t& p0) {
  if (a.items) {
    const FusedItem w = a.items[it];
    inst = w.inst;
    p0 = (int64_t)w.tile * TM;
  } else {
    inst = 0;
    p0 = it * TM;
  }
}

// -(1024 2^-K + OFFSET) in both halves: a multiple of its last place, exact.
__host__ __device__ constexpr uint32_t minus_of(int K, uint32_t offset) { return (0x8000u | ((25u - K) << 10) | (offset << K)) * 0x10001u; }
__device__ __forceinline__ void fill_digit_const(DigitConst& c) {
  c.pattern = 0x64006400u;
  c.mask7 = 0x007f007fu;
  c.mask6 = 0x003f003fu;
  c.mask6_2 = 0x00fc00fcu;
  c.mask6_4 = 0x03f003f0u;
  c.minus7 = minus_of(0, 64);
  c.minus6 = minus_of(0, 32);
  c.minus6_2 = minus_of(2, 32);
  c.minus6_4 = minus_of(4, 32);
  c.scale_2 = 0x34003400u;  // 1 / 4
  c.scale_4 = 0x2c002c00u;  // 1 / 16
}
// One digit of two words as two float16: a byte permute brings a 16-bit window holding the field
// (0, 2 or 4 bits up) of each word together, the mask and the pattern make 1024 + field 2^K, and one
// packed (multiply-)add takes off the offset and the 2^K (all exact).
__device__ __forceinline__ uint32_t digit_at0(uint32_t window, uint32_t mask, uint32_t minus, const DigitConst& c) {
  const uint32_t w = (window & mask) | c.pattern;
  const __half2 v = __hadd2(*reinterpret_cast<const __half2*>(&w), *reinterpret_cast<const __half2*>(&minus));
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ uint32_t digit_up(uint32_t window, uint32_t mask, uint32_t scale, uint32_t minus,
                                             const DigitConst& c) {
  const uint32_t w = (window & mask) | c.pattern;
  const __half2 v = __hfma2(*reinterpret_cast<const __half2*>(&w), *reinterpret_cast<const __half2*>(&scale),
                            *reinterpret_cast<const __half2*>(&minus));
  return *reinterpret_cast<const uint32_t*>(&v);
}

// The nine digits of two words (x low), each two float16.  Leading field at bits 56-62, then six
// bits each downwards to bit 8: no field crosses the word's middle.
__device__ __forceinline__ void digits_of(uint64_t x, uint64_t y, uint32_t (&w)[TND], const DigitConst& c) {
  const uint32_t xh = (uint32_t)(x >> 32), yh = (uint32_t)(y >> 32), xl = (uint32_t)x, yl = (uint32_t)y;
  auto up2 = [&](uint32_t v) { return digit_up(v, c.mask6_2, c.scale_2, c.minus6_2, c); };
  auto up4 = [&](uint32_t v) { return digit_up(v, c.mask6_4, c.scale_4, c.minus6_4, c); };
  w[0] = digit_at0(__byte_perm(xh, yh, 0x7733), c.mask7, c.minus7, c);
  w[1] = up2(__byte_perm(xh, yh, 0x6622));
  w[2] = up4(__byte_perm(xh, yh, 0x6521));
  const uint32_t low_h = __byte_perm(xh, yh, 0x5410);
  w[3] = up4(low_h >> 2);
  w[4] = digit_at0(low_h, c.mask6, c.minus6, c);
  w[5] = up2(__byte_perm(xl, yl, 0x7733));
  w[6] = up4(__byte_perm(xl, yl, 0x7632));
  const uint32_t mid_l = __byte_perm(xl, yl, 0x6521);
  w[7] = up4(mid_l >> 2);
  w[8] = digit_at0(mid_l, c.mask6, c.minus6, c);
}

// Stores a chunk's digits: digit t in columns 8 t .. 8 t + 3 from `at` (this half's four).
template <int T = 0>
__device__ __forceinline__ void store_digits(uint32_t at, const uint32_t (&e0)[TND], const uint32_t (&e1)[TND],
                                             const uint32_t (&o0)[TND], const uint32_t (&o1)[TND]) {
  if constexpr (T < TND) {
    ptx::tmem_st_32x32b_x4<8 * T>(at, e0[T], e1[T], o0[T], o1[T]);
    store_digits<T + 1>(at, e0, e1, o0, o1);
  }
}

// A finished segment of this thread's tile, kept until it is drained.
struct Pending {
  int inst = -1, ep = 0;
  bool first = true;     // the tile's first segment
  int64_t p0 = 0;
  double c = 1.0, s = 0.0, rho = 0.0;  // gradients: the point's angle and radius
};

// Out of line: sixteen inlined copies would not fit the instruction cache beside the walk.
__device__ __noinline__ double join_rounded(long long hi, long long lo, int ls, int e2) {
  return join_to_double(hi, lo, ls, e2);
}

// Drains the accumulators of a finished segment for this thread's row and 8 sets: per set nine
// diagonal sums out of tensor memory, recombined exactly and rounded once to float64.
template <int GROUPS>
__device__ __forceinline__ bool drain_segment(const TriArgs& a, const Pending& pd, uint32_t tmem_base, uint32_t acc,
                                              uint32_t quad, int lane, int half, double* swap, Barriers* bar,
                                              uint32_t parity) {
  const TriInst& d = inst_of(a, pd.inst);
  const int64_t p = pd.p0 + quad * 32 + lane;
  constexpr int Split = 4;
  double dot[2] = {0.0, 0.0};
#pragma unroll
  for (int g = 0; g < GROUPS; ++g) {
    long long hi[8] = {}, lo[8] = {};
#pragma unroll
    for (int db = 0; db < TND; ++db) {
      const int block = g == 1 ? TND - 1 - db : db;
      uint32_t v[8];
      ptx::tmem_ld_32x32b_x8(
          tmem_base + ((quad * 32u) << 16) + (GROUPS == 2 ? (uint32_t)g : acc) * kAccCols + (uint32_t)(block * TNS + half * 8), v);
      ptx::tmem_ld_wait(v);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const long long tv = (long long)__float2int_rn(__uint_as_float(v[i]));
        if (db < Split) hi[i] = horner(hi[i], 6, tv);
        else lo[i] = horner(lo[i], 6, tv);
      }
    }
    const int e_base = pd.ep - 6 * (TND + 1);
    const int* cexp = d.cexp + g * TNS;
    if (p < d.P) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int s = half * 8 + i;
        if (s >= d.S) break;
        const int ec = cexp[s];
        const double v = (pd.ep == kNonFiniteRow || ec == kNonFiniteRow)
                             ? __longlong_as_double(0x7ff8000000000000ll)
                             : join_rounded(hi[i], lo[i], 6 * (TND - Split), e_base + ec);
        if constexpr (GROUPS == 2) {
          dot[g] = fma(d.gdot[p * d.S + s], v, dot[g]);
        } else {
          double* o = d.out + p * d.S + s;
          *o = pd.first ? v : *o + v;
        }
      }
    }
    // All lanes take the next tensor-memory load together: those beyond the last point, and those that
    // join_rounded parted, meet here.
    __syncwarp();
  }
  if constexpr (GROUPS == 2) {
    // The two halves' sums of a point meet in shared memory.
    double* mine = swap + quad * 32 + lane;
    if (half == 1) {
      mine[0] = dot[0];
      mine[TM] = dot[1];
    }
    if (half == 1) {
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&bar->swap_full[quad]);
      if (!warp_wait(&bar->swap_empty[quad], parity, &bar->abort_flag, lane)) return false;
    } else {
      if (!warp_wait(&bar->swap_full[quad], parity, &bar->abort_flag, lane)) return false;
      const double dx = dot[0] + mine[0], dy = dot[1] + mine[TM];
      if (p < d.P) {
        const double gr = fma(pd.c, dx, pd.s * dy), gt = pd.rho * fma(pd.c, dy, -pd.s * dx);
        if (d.grad_r) d.grad_r[p] = pd.first ? gr : d.grad_r[p] + gr;
        if (d.grad_theta) d.grad_theta[p] = pd.first ? gt : d.grad_theta[p] + gt;
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&bar->swap_empty[quad]);
    }
  }
  return true;
}

// A chunk's digits from values walked in float64, digitised at the row's scale.  Out of line, so that the
// fixed-point digits' registers and code are not laid out around it: 1e6 points on the disc, n <= 32, 16 sets
// 2.41 -> 2.32 ms; a 1000 x 1000 pixel grid with a fifth of its points off the disc 4.29 -> 4.46 ms.
__device__ __noinline__ void digits_of_float64(const uint64_t* f, const ulonglong2* an, TriBlock bi, int n_max, bool zero_row,
                                               int shift, uint32_t at, DigitConst dc) {
  const int H = n_max / 2;
#pragma unroll 1
  for (int k = 0; k < 2; ++k) {
    const TriAngleRows am = tri_angle_rows(2 * (bi.A - bi.B), n_max);
    const int n0 = 2 * (bi.A + bi.B);
    uint32_t w[4][TND];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint64_t y[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int n = n0 + (e == 0 ? 0 : e == 3 ? 2 : 1);
        const ulonglong2 g = an[(size_t)(e == 1 ? am.low : e == 2 ? am.top : am.mid) * TM];
        const double z = __longlong_as_double((long long)f[(size_t)(4 * k + e) * TM]) *
                         __longlong_as_double((long long)(h ? g.y : g.x));
        // Elements above n_max (and all of a non-finite row) have no coefficients: zero.
        y[e] = (uint64_t)(zero_row || n > n_max ? 0 : to_fixed(z, shift)) + kTriWordBias;
      }
      digits_of(y[0], y[1], w[2 * h], dc);
      digits_of(y[2], y[3], w[2 * h + 1], dc);
    }
    __syncwarp();  // to_fixed parts the lanes; a tensor-memory store is the whole warp's
    store_digits(at + 4u * k, w[0], w[1], w[2], w[3]);
    bi.advance(H);
  }
}

// Row scale exponent of a point walked in float64: 2^E above 1.02 times the largest |R| of its
// triangle (the margin keeps the leading digit's field within seven bits); kNonFiniteRow when a
// value is not finite.
__device__ __forceinline__ int scale_of(double most) {
  if (!isfinite(most)) return kNonFiniteRow;
  const double wide = most * 1.02;
  return isfinite(wide) ? scale_exponent((unsigned long long)__double_as_longlong(wide)) : 1024;
}
// n_max <= 3 (tiles of one chunk): the polynomials themselves, for the digit warps too.
__device__ __forceinline__ int row_scale_low(double rho, int n_max) {
  if (!isfinite(rho)) return kNonFiniteRow;  // also of n_max = 0, which has no polynomial of rho below
  double most = 1.0;
  const double u = rho * rho, R[5] = {rho, fma(2.0, u, -1.0), u, rho * fma(3.0, u, -2.0), rho * u};
  const int n_of[5] = {1, 2, 2, 3, 3};
  for (int i = 0; i < 5; ++i)
    if (n_of[i] <= n_max && !(fabs(R[i]) <= most)) most = fabs(R[i]);
  return scale_of(most);
}
// Otherwise a first walk (walk warps; st: the row's state).
__device__ __noinline__ int row_scale(double rho, int n_max, uint64_t* st) {
  double most = 0.0;
  const int H = n_max / 2;
  auto note = [&](double f, int n) {
    if (n <= n_max && !(fabs(f) <= most)) most = fabs(f);
  };
  for (int A = 0; A <= H; ++A) {
    const int nb = min(A, H - A);
    double l0 = 0.0, l1 = 0.0, dg = A == 0 ? -1.0 : 0.0;
    for (int B = 0; B <= nb && most <= 1.7e308; ++B) {
      uint64_t* row = st + (size_t)(2 * B) * TM;
      const double u0 = B < A ? __longlong_as_double((long long)row[0]) : l0;
      const double u1 = B < A ? __longlong_as_double((long long)row[TM]) : l1;
      const double e00 = fma(rho, u0 + l0, -dg), e01 = fma(rho, u1 + e00, -u0);
      const double e10 = fma(rho, e00 + l1, -l0), e11 = fma(rho, e01 + e10, -e00);
      row[0] = (uint64_t)__double_as_longlong(e10);
      row[TM] = (uint64_t)__double_as_longlong(e11);
      dg = u1;
      l0 = e01;
      l1 = e11;
      const int n0 = 2 * (A + B);
      note(e00, n0);
      note(e01, n0 + 1);
      note(e10, n0 + 1);
      note(e11, n0 + 2);
    }
  }
  return scale_of(most);
}

// Rows m0 .. m1 - 1 of the angle table: (cos, sin) entries of the fixed-point walk.
__device__ __forceinline__ void fill_angles(ulonglong2* an, uint64_t turn, int64_t ci, int64_t si, int m0, int m1) {
  const TriTrig c1 = tri_split(ci), s1 = tri_split(si);
  TriTrig c = tri_split(1ll << 62), s = tri_split(0);
  if (m0 > 0) {
    int64_t cm, sm;
    tri_cos_sin(turn * (uint64_t)m0, cm, sm);
    c = tri_split(cm);
    s = tri_split(sm);
  }
  for (int m = m0; m < m1; ++m) {
    an[(size_t)m * TM] = make_ulonglong2(tri_entry(c), tri_entry(s));
    tri_rotate(c, s, c1, s1);
  }
}
// The same as float64 cos and sin, by angle addition.
__device__ __noinline__ void fill_angles_f64(ulonglong2* an, double c1, double s1, int m0, int m1) {
  double c = 1.0, s = 0.0;
  for (int m = 0; m < m1; ++m) {
    if (m >= m0)
      an[(size_t)m * TM] = make_ulonglong2((uint64_t)__double_as_longlong(c), (uint64_t)__double_as_longlong(s));
    const double cn = fma(c, c1, -s * s1);
    s = fma(s, c1, c * s1);
    c = cn;
  }
}

template <int GROUPS>
__global__ void __launch_bounds__(kThreads, 1) tri_kernel(TriArgs a, int n_max_launch, int n_stages) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 255) & ~uintptr_t(255));
  constexpr uint32_t kStageB = stage_bytes(GROUPS);
  constexpr uint32_t kZeroAt = GROUPS == 2 ? kTriGroupBytes : 0;  // zero blocks of a stage
  uint8_t* rest = smem + (uint32_t)n_stages * kStageB;
  Barriers* bar = reinterpret_cast<Barriers*>(rest);
  uint64_t* ring = reinterpret_cast<uint64_t*>(rest + kAux);                   // [slot][8][row]
  int* ring_scale = reinterpret_cast<int*>(rest + kAux + kRing * kSlotB);      // [slot][row], float64 walks
  ulonglong2* angles = reinterpret_cast<ulonglong2*>(rest + kAux + kRingB);    // [m][row]
  uint64_t* state = reinterpret_cast<uint64_t*>(rest + kAux + kRingB + angle_bytes(n_max_launch));  // [b][row]
  double* swap = reinterpret_cast<double*>(rest + kAux + kRingB + angle_bytes(n_max_launch) + state_bytes(n_max_launch));
  volatile int* abort_flag = &bar->abort_flag;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      ptx::mbar_init(&bar->full[i], 4);
      ptx::mbar_init(&bar->empty[i], 1);
    }
    for (int i = 0; i < kMaxBStages; ++i) {
      ptx::mbar_init(&bar->bfull[i], 1);
      ptx::mbar_init(&bar->bempty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&bar->tfull[i], 1);
      ptx::mbar_init(&bar->tempty[i], kDigitWarps);
    }
    for (int i = 0; i < 4; ++i) {
      for (int j = 0; j < kRing; ++j) {
        ptx::mbar_init(&bar->rfull[j][i], 1);
        ptx::mbar_init(&bar->rempty[j][i], 1);
      }
      ptx::mbar_init(&bar->table_ready[i], 2);
      ptx::mbar_init(&bar->table_free[i], 2);
      ptx::mbar_init(&bar->swap_full[i], 1);
      ptx::mbar_init(&bar->swap_empty[i], 1);
    }
    ptx::mbar_init(&bar->drain, 1);
    bar->abort_flag = 0;
    fill_digit_const(bar->digits);
    ptx::fence_barrier_init();
  }
  for (uint32_t i = threadIdx.x; i < (uint32_t)n_stages * kZeroB / 16; i += kThreads) {
    const uint32_t st = i / (kZeroB / 16), o = i % (kZeroB / 16);
    reinterpret_cast<uint4*>(smem + st * kStageB + kZeroAt)[o] = make_uint4(0u, 0u, 0u, 0u);
  }
  ptx::fence_proxy_async_smem();
  if (warp == kMmaWarp) {
    ptx::tmem_alloc(&bar->tmem_base, kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = bar->tmem_base;
  const uint32_t quad = (uint32_t)(warp & 3);
  const uint32_t row = quad * 32 + lane;  // point row of the tile (digit and walk warps)

  // This row's point and whether its quadrant walks in float64 (digit and walk warps agree).
  auto point_of = [&](const TriInst& d, int64_t p0, double& rho, double& th) -> bool {
    const int64_t p = p0 + row;
    const bool valid = p < d.P;
    rho = valid ? d.r[p] : 0.0;
    th = valid && d.theta ? d.theta[p] : 0.0;
    const uint32_t e = ((uint32_t)__double2hiint(th) >> 20) & 0x7ffu;
    return __any_sync(0xffffffffu, !(rho >= 0.0 && rho <= 1.0 && e < (uint32_t)kTriAngleExponent));
  };

  if (warp < kDigitWarps) {
    // ------------------------------------------------------------ digits (and accumulator drain)
    const int group = warp >> 2;
    ulonglong2* an = angles + row;
    int stage = 0, slot = 0;
    uint32_t sphase = 0, rphase = 0;
    int turn_of = 0;         // the group that takes the next chunk
    uint32_t n_drained = 0;  // segments drained
    uint32_t tile = 0;
    const DigitConst dc = bar->digits;
    bool ok = true;
    Pending prev;
    auto drain_prev = [&]() {
      const uint32_t acc = GROUPS == 2 ? 0u : n_drained & 1u, use = GROUPS == 2 ? n_drained & 1u : (n_drained >> 1) & 1u;
      ok = warp_wait(&bar->tfull[acc], use, abort_flag, lane);
      if (!ok) return;
      ptx::tc_fence_after();
      ok = drain_segment<GROUPS>(a, prev, tmem_base, acc, quad, lane, group, swap, bar, n_drained & 1u);
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&bar->tempty[acc]);
      ++n_drained;
      prev.inst = -1;
    };
    for (int64_t it = blockIdx.x; it < a.n_items && ok; it += gridDim.x, ++tile) {
      int ii;
      int64_t p0;
      item_of(a, it, ii, p0);
      const TriInst& d = inst_of(a, ii);
      const int n_max = d.n_max, H = n_max / 2, KC = d.KC, seg_chunks = d.seg_chunks;
      double rho, th;
      const bool slow = point_of(d, p0, rho, th);
      Pending cur;
      cur.inst = ii;
      cur.p0 = p0;
      cur.ep = 1;
      cur.rho = rho;

      bool zero_row = false;  // float64 walk: a non-finite row, and the row's scale
      int shift = 0;
      auto set_scale = [&](int E) {
        zero_row = E == kNonFiniteRow || !isfinite(th);
        cur.ep = zero_row ? kNonFiniteRow : E;
        shift = kRowScale - (zero_row ? 0 : E);
      };

      // The quadrant's angle table, half of it by each of its two warps.
      if (tile > 0) {
        ok = warp_wait(&bar->table_free[quad], (tile - 1) & 1u, abort_flag, lane);
        if (!ok) break;
      }
      const int mid_row = (n_max + 2) / 2, from = group ? mid_row : 0, to = group ? n_max + 1 : mid_row;
      if (!slow) {
        const uint64_t turn = tri_turn((uint64_t)__double_as_longlong(th));
        int64_t ci, si;
        tri_cos_sin(turn, ci, si);
        if constexpr (GROUPS == 2) {
          cur.c = (double)ci * 0x1p-62;
          cur.s = (double)si * 0x1p-62;
        }
        fill_angles(an, turn, ci, si, from, to);
      } else {
        if (KC == 1) set_scale(row_scale_low(rho, n_max));
        sincos(th, &cur.s, &cur.c);
        fill_angles_f64(an, cur.c, cur.s, from, to);
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&bar->table_ready[quad]);
      ok = warp_wait(&bar->table_ready[quad], tile & 1u, abort_flag, lane);
      if (!ok) break;
      if constexpr (GROUPS == 2) {
        if (prev.inst >= 0) drain_prev();
        if (!ok) break;
      }

      const uint32_t lane_base = tmem_base + ((quad * 32u) << 16) + kABase;
      TriBlock bi;
      int seg_left = seg_chunks;
      for (int kc = 0; kc < KC; ++kc) {
        if (turn_of == group) {
          const uint64_t* f = ring + (size_t)slot * 8 * TM + row;
          ok = warp_wait(&bar->rfull[slot][quad], rphase, abort_flag, lane);
          if (!ok) break;
          if (!slow) {
            // Straight-line code for the chunk's two blocks, so that the second one's products
            // overlap the first one's digits.
            uint64_t v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = f[(size_t)k * TM];
            ok = warp_wait(&bar->empty[stage], sphase ^ 1u, abort_flag, lane);
            if (!ok) break;
            ptx::tc_fence_after();
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const TriAngleRows am = tri_angle_rows(2 * (bi.A - bi.B), n_max);
              const ulonglong2 mid = an[(size_t)am.mid * TM], low = an[(size_t)am.low * TM], top = an[(size_t)am.top * TM];
              uint32_t wc0[TND], wc1[TND], ws0[TND], ws1[TND];
              const uint64_t mc = tri_offset(mid.x), ms = tri_offset(mid.y);
              digits_of(tri_word(v[4 * k], mid.x, mc), tri_word(v[4 * k + 1], low.x, tri_offset(low.x)), wc0, dc);
              digits_of(tri_word(v[4 * k + 2], top.x, tri_offset(top.x)), tri_word(v[4 * k + 3], mid.x, mc), wc1, dc);
              digits_of(tri_word(v[4 * k], mid.y, ms), tri_word(v[4 * k + 1], low.y, tri_offset(low.y)), ws0, dc);
              digits_of(tri_word(v[4 * k + 2], top.y, tri_offset(top.y)), tri_word(v[4 * k + 3], mid.y, ms), ws1, dc);
              store_digits(lane_base + (uint32_t)stage * kAStage + 4u * k, wc0, wc1, ws0, ws1);
              bi.advance(H);
            }
          } else {
            // Values walked in float64, digitised at the row's scale (each group takes at least one
            // chunk of a tile of several, and so learns it).
            if (KC > 1) set_scale(ring_scale[slot * TM + row]);
            ok = warp_wait(&bar->empty[stage], sphase ^ 1u, abort_flag, lane);
            if (!ok) break;
            ptx::tc_fence_after();
            digits_of_float64(f, an, bi, n_max, zero_row, shift, lane_base + (uint32_t)stage * kAStage, dc);
            bi.advance(H);
            bi.advance(H);
          }
          ptx::tmem_st_wait();
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            ptx::mbar_arrive(&bar->rempty[slot][quad]);
            ptx::mbar_arrive(&bar->full[stage]);
          }
        } else {
          bi.advance(H);
          bi.advance(H);
        }
        turn_of ^= 1;
        if (++stage == kStages) {
          stage = 0;
          sphase ^= 1u;
        }
        if (++slot == kRing) {
          slot = 0;
          rphase ^= 1u;
        }
        if (--seg_left == 0 || kc == KC - 1) {
          if (kc == KC - 1) {
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&bar->table_free[quad]);
          }
          if (GROUPS == 1 && prev.inst >= 0) drain_prev();
          prev = cur;
          cur.first = false;
          seg_left = seg_chunks;
          // Two groups use both accumulators: this segment leaves them before the next begins.
          if (GROUPS == 2 && kc < KC - 1 && ok) drain_prev();
          if (!ok) break;
        }
      }
      if (!ok) break;
    }
    if (ok && prev.inst >= 0) drain_prev();
    if (!ok) fail(abort_flag);
  } else if (warp < kMmaWarp) {
    // ------------------------------------------------------------ the radial walk
    uint64_t* st = state + row;
    int slot = 0;
    uint32_t rphase = 0;
    bool ok = true;
    for (int64_t it = blockIdx.x; it < a.n_items && ok; it += gridDim.x) {
      int ii;
      int64_t p0;
      item_of(a, it, ii, p0);
      const TriInst& d = inst_of(a, ii);
      const int n_max = d.n_max, H = n_max / 2, KC = d.KC;
      double rho, th;
      const bool slow = point_of(d, p0, rho, th);
      const TriPoint tp = tri_point((uint64_t)__double_as_longlong(rho));
      const int scale = slow && KC > 1 ? row_scale(rho, n_max, st) : 0;
      TriBlock bi;
      uint64_t l0 = 0, l1 = 0, dg = 0;  // f(2A, 2B-1), f(2A+1, 2B-1), f(2A-1, 2B-1): biased words or float64 bits
      for (int kc = 0; kc < KC; ++kc) {
        ok = warp_wait(&bar->rempty[slot][quad], rphase ^ 1u, abort_flag, lane);
        if (!ok) break;
        uint64_t* f = ring + (size_t)slot * 8 * TM + row;
        if (!slow) {
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const bool begin = bi.B == 0, diag = bi.B == bi.A;
            uint64_t* r = st + (size_t)(2 * bi.B) * TM;
            const uint64_t s0 = r[0], s1 = r[TM];
            l0 = begin ? kTriZero : l0;
            l1 = begin ? kTriZero : l1;
            dg = begin ? (bi.A == 0 ? 0ull : kTriZero) : dg;
            const uint64_t u0 = diag ? l0 : s0, u1 = diag ? l1 : s1;
            const uint64_t e00 = tri_floor(tri_step(tp, u0, l0, dg)), e01 = tri_step(tp, u1, e00, u0);
            const uint64_t e10 = tri_step(tp, e00, l1, l0), e11 = tri_floor(tri_step(tp, e01, e10, e00));
            r[0] = e10;
            r[TM] = e11;
            f[(size_t)(4 * k) * TM] = e00;
            f[(size_t)(4 * k + 1) * TM] = e01;
            f[(size_t)(4 * k + 2) * TM] = e10;
            f[(size_t)(4 * k + 3) * TM] = e11;
            dg = u1;
            l0 = e01;
            l1 = e11;
            bi.advance(H);
          }
        } else {
          ring_scale[slot * TM + row] = scale;
#pragma unroll 1
          for (int k = 0; k < 2; ++k) {
            const bool begin = bi.B == 0, diag = bi.B == bi.A;
            uint64_t* r = st + (size_t)(2 * bi.B) * TM;
            auto f64 = [](uint64_t v) { return __longlong_as_double((long long)v); };
            auto bits = [](double v) { return (uint64_t)__double_as_longlong(v); };
            const double f_l0 = begin ? 0.0 : f64(l0), f_l1 = begin ? 0.0 : f64(l1);
            const double f_dg = begin ? (bi.A == 0 ? -1.0 : 0.0) : f64(dg);
            const double u0 = diag ? f_l0 : f64(r[0]), u1 = diag ? f_l1 : f64(r[TM]);
            const double e00 = fma(rho, u0 + f_l0, -f_dg), e01 = fma(rho, u1 + e00, -u0);
            const double e10 = fma(rho, e00 + f_l1, -f_l0), e11 = fma(rho, e01 + e10, -e00);
            r[0] = bits(e10);
            r[TM] = bits(e11);
            f[(size_t)(4 * k) * TM] = bits(e00);
            f[(size_t)(4 * k + 1) * TM] = bits(e01);
            f[(size_t)(4 * k + 2) * TM] = bits(e10);
            f[(size_t)(4 * k + 3) * TM] = bits(e11);
            dg = bits(u1);
            l0 = bits(e01);
            l1 = bits(e11);
            bi.advance(H);
          }
        }
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&bar->rfull[slot][quad]);
        if (++slot == kRing) {
          slot = 0;
          rphase ^= 1u;
        }
      }
    }
    if (!ok) fail(abort_flag);
  } else if (warp == kMmaWarp) {
    // The whole warp runs the loop and one lane issues: with warp-uniform control flow (votes,
    // warp reductions of the loaded values) the operands stay in uniform registers, where one
    // thread's loop spent most of its time moving them there (1.9 of 2.5 million cycles).
    constexpr uint32_t kAll = 0xffffffffu;
    constexpr uint32_t idesc = ptx::idesc_f16_f32(TM, kAccCols);
    const uint32_t tmem = __reduce_max_sync(kAll, tmem_base);
    const uint64_t desc0 = ptx::sw_kmajor_desc<kRowB>(0) + (ptx::smem_u32(smem) >> 4);
    int stage = 0, bstage = 0;
    uint32_t phase = 0, bphase = 0, n_segs = 0;
    bool ok = true;
    for (int64_t it = blockIdx.x; it < a.n_items && ok; it += gridDim.x) {
      int ii;
      int64_t p0;
      item_of(a, it, ii, p0);
      const TriInst& d = inst_of(a, ii);
      const int KC = (int)__reduce_max_sync(kAll, (unsigned)d.KC);
      const int seg_chunks = (int)__reduce_max_sync(kAll, (unsigned)d.seg_chunks);
      for (int kc0 = 0; kc0 < KC && ok; kc0 += seg_chunks, ++n_segs) {
        const uint32_t acc = GROUPS == 2 ? 0u : n_segs & 1u, use = GROUPS == 2 ? n_segs & 1u : (n_segs >> 1) & 1u;
        ok = __all_sync(kAll, ptx::mbar_wait(&bar->tempty[acc], use ^ 1u, abort_flag));
        if (!ok) break;
        ptx::tc_fence_after();
        const int kc1 = min(KC, kc0 + seg_chunks);
        for (int kc = kc0; kc < kc1; ++kc) {
          ok = __all_sync(kAll, ptx::mbar_wait(&bar->full[stage], phase, abort_flag) &&
                                    ptx::mbar_wait(&bar->bfull[bstage], bphase, abort_flag));
          if (!ok) break;
          ptx::tc_fence_after();
          const uint64_t bd = desc0 + (uint32_t)bstage * (kStageB >> 4);
          const uint32_t at = tmem + kABase + (uint32_t)stage * kAStage;
          const uint32_t accumulate = kc == kc0 ? 0u : 1u;
          if (lane == 0) {
#pragma unroll
            for (int t = 0; t < TND; ++t) {
              const uint32_t more = t == 0 ? accumulate : 1u;
              if constexpr (GROUPS == 1) {
                // Coefficient blocks shifted down by t: diagonal t + u receives a_t b_u.
                ptx::mma_f16_tmem_a(tmem + acc * kAccCols, at + t * 8, bd + (TND - 1 - t) * (kBlockB >> 4), idesc, more);
              } else {
                ptx::mma_f16_tmem_a(tmem, at + t * 8, bd + (2 * TND - 1 - t) * (kBlockB >> 4), idesc, more);
                ptx::mma_f16_tmem_a(tmem + kAccCols, at + t * 8, bd + t * (kBlockB >> 4), idesc, more);
              }
            }
            ptx::mma_commit(&bar->empty[stage]);
            ptx::mma_commit(&bar->bempty[bstage]);
          }
          __syncwarp();
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1u;
          }
          if (++bstage == n_stages) {
            bstage = 0;
            bphase ^= 1u;
          }
        }
        if (ok && lane == 0) ptx::mma_commit(&bar->tfull[acc]);
        __syncwarp();
      }
    }
    if (lane == 0) {
      if (!ok) fail(abort_flag);
      // Every MMA this thread issued has completed before TMEM is released (a wait that ignores
      // the abort flag, still bounded).
      ptx::mma_commit(&bar->drain);
      int never = 0;
      if (!ptx::mbar_wait(&bar->drain, 0u, &never)) atomicOr(&g_tri_error, 1u);
    }
    __syncwarp();
  } else if (lane == 0) {
    // Coefficient copies, one chunk per stage.
    int stage = 0;
    uint32_t phase = 0;
    uint32_t issued[kMaxBStages] = {};
    bool ok = true;
    for (int64_t it = blockIdx.x; it < a.n_items && ok; it += gridDim.x) {
      int ii;
      int64_t p0;
      item_of(a, it, ii, p0);
      const TriInst& d = inst_of(a, ii);
      const int KC = d.KC;
      for (int kc = 0; kc < KC; ++kc) {
        if (!ptx::mbar_wait(&bar->bempty[stage], phase ^ 1u, abort_flag)) {
          ok = false;
          break;
        }
        uint8_t* dst = smem + (uint32_t)stage * kStageB;
        const uint8_t* src = d.bdig + (size_t)kc * (GROUPS * kTriGroupBytes);
        ptx::mbar_arrive_expect_tx(&bar->bfull[stage], GROUPS * kTriGroupBytes);
        if constexpr (GROUPS == 1) {
          ptx::bulk_g2s(dst + kZeroB, src, kTriGroupBytes, &bar->bfull[stage]);
        } else {
          ptx::bulk_g2s(dst + kZeroB + kTriGroupBytes, src, kTriGroupBytes, &bar->bfull[stage]);
          ptx::bulk_g2s(dst, src + kTriGroupBytes, kTriGroupBytes, &bar->bfull[stage]);
        }
        for (int i = 0; i < kMaxBStages; ++i) issued[i] += i == stage;
        if (++stage == n_stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok) fail(abort_flag);
    // Every copy has landed before the CTA may exit (ignoring the abort flag, still bounded).
    int never = 0;
    for (int i = 0; i < kMaxBStages; ++i)
      if (issued[i] && !ptx::mbar_wait(&bar->bfull[i], (issued[i] - 1u) & 1u, &never)) atomicOr(&g_tri_error, 1u);
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, kTmemCols);
  }
}

// Instance and chunk of block `g` of a launch over all chunks.
__device__ __forceinline__ const TriInst& chunk_of(const TriArgs& a, const int32_t* chunk_inst, int64_t g, int64_t& kc) {
  const TriInst& d = inst_of(a, chunk_inst ? chunk_inst[g] : 0);
  kc = g - d.kc_base;
  return d;
}

// Coefficients of dF/dx and dF/dy over the triangle (see the top of the file): with
// C = alpha (cos) and beta (sin) of degree n, A_l^m = sum_{n >= l, n = l mod 2} alpha_n^m and B
// likewise, position (l, m) holds for x  (l+1) (A_{l+1}^{m+1} + A_{l+1}^{m-1}) cos and the same of
// B for sin, for y  (l+1) (B^{m+1} - B^{m-1}) cos and -(l+1) (A^{m+1} - A^{m-1}) sin; at m = 1 the
// m - 1 = 0 term counts twice, at m = 0 there is none.  One block per chunk, thread = (position,
// set); cpos [2][chunks * 16][16].
__global__ void __launch_bounds__(kTriChunk * TNS) tri_deriv_kernel(TriArgs a, const int32_t* chunk_inst) {
  int64_t kc;
  const TriInst& d = chunk_of(a, chunk_inst, blockIdx.x, kc);
  const int s = threadIdx.x % TNS;
  const int pos = (int)kc * kTriChunk + threadIdx.x / TNS;
  int n, m, sine;
  tri_mode(pos, d.n_max, n, m, sine);
  // A set with coefficients near the top of the range is formed 2^-24 down (the sums below grow by at most
  // (n + 1) 96 < 2^13), which its scale takes up again.
  __shared__ int high[TNS];
  if (threadIdx.x < TNS) high[threadIdx.x] = 0;
  __syncthreads();
  if (s < d.S) {
    bool top = false;
#pragma unroll 8
    for (int64_t j = threadIdx.x / TNS; j < d.J; j += kTriChunk) top |= !(fabs(d.coeffs[j * d.S + s]) < 0x1p1000);
    if (top) high[s] = 1;
  }
  __syncthreads();
  const int down = high[s] ? 24 : 0;
  const double scale = down ? 0x1p-24 : 1.0;
  if (kc == 0 && threadIdx.x < TNS) d.cexp[s] = d.cexp[TNS + s] = down;  // tri_coeff_kernel adds the rest
  double vx = 0.0, vy = 0.0;
  if (s < d.S && m >= 0 && n < d.n_max && !(m == 0 && sine)) {
    // Sums over n' = n + 1, n + 3, .. of the coefficients of (n', mm), cos or sin.
    auto sum = [&](int mm, int h) {
      double t = 0.0;
      if (mm < 0 || (mm == 0 && h)) return t;
      for (int k = n + 1; k <= d.n_max; k += 2) {
        if (mm > k) continue;
        const int32_t j = __ldg(d.perm + tri_position(k, mm, h, d.n_max));
        if (j >= 0) t = fma(scale, d.coeffs[(int64_t)j * d.S + s], t);
      }
      return t;
    };
    const double f = (double)(n + 1), twice = m == 1 ? 2.0 : 1.0;
    if (sine == 0) {
      vx = f * (sum(m + 1, 0) + (m > 0 ? twice * sum(m - 1, 0) : 0.0));
      vy = f * (sum(m + 1, 1) - (m > 0 ? twice * sum(m - 1, 1) : 0.0));
    } else {
      vx = f * (sum(m + 1, 1) + twice * sum(m - 1, 1));
      vy = -f * (sum(m + 1, 0) - twice * sum(m - 1, 0));
    }
  }
  const int64_t total = (int64_t)d.KC * kTriChunk;
  d.cpos[(int64_t)pos * TNS + s] = vx;
  d.cpos[(total + pos) * TNS + s] = vy;
}

// Coefficient digits of one chunk and group (blockIdx.y): the sets' scales 2^e > max |C| (formed by
// every block from all of the group's coefficients; the first chunk's block stores them, with what
// tri_deriv_kernel took off), then
// 9 digits per coefficient as float16 rows of 32 bytes (32-byte swizzle), the second group's
// blocks in reverse order.
__global__ void __launch_bounds__(kTriChunk * TNS) tri_coeff_kernel(TriArgs a, const int32_t* chunk_inst) {
  __shared__ unsigned long long red[kTriChunk][TNS];
  int64_t kc;
  const TriInst& d = chunk_of(a, chunk_inst, blockIdx.x, kc);
  const int g = blockIdx.y, groups = gridDim.y;
  const int s = threadIdx.x % TNS, q = threadIdx.x / TNS;
  const int64_t total = (int64_t)d.KC * kTriChunk;
  const double* src = d.cpos ? d.cpos + g * total * TNS : nullptr;
  unsigned long long mx = 0;
  if (s < d.S) {
    const int64_t rows = src ? total : d.J, stride = src ? TNS : d.S;
    const double* base = src ? src : d.coeffs;
#pragma unroll 8
    for (int64_t j = q; j < rows; j += kTriChunk) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(base[j * stride + s]) & 0x7fffffffffffffffull;
      mx = b > mx ? b : mx;
    }
  }
  red[q][s] = mx;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kTriChunk; ++i) mx = red[i][s] > mx ? red[i][s] : mx;
  const int ec = scale_exponent(mx);
  if (kc == 0 && q == 0) d.cexp[g * TNS + s] = ec + (src && ec != kNonFiniteRow ? d.cexp[g * TNS + s] : 0);
  const int64_t pos = kc * kTriChunk + q;
  double c = 0.0;
  if (s < d.S && ec != kNonFiniteRow) {
    if (src) {
      c = src[pos * TNS + s];
    } else {
      const int32_t j = __ldg(d.perm + pos);
      if (j >= 0) c = d.coeffs[(int64_t)j * d.S + s];
    }
  }
  long long y = c == 0.0 ? 0 : to_fixed(c, 6 * TND - ec);
#pragma unroll
  for (int k = 0; k < TND - 1; ++k) y += 32ll << (6 * k);
  uint8_t* chunk = d.bdig + ((size_t)kc * groups + g) * kTriGroupBytes;
#pragma unroll
  for (int t = 0; t < TND; ++t) {
    const int digit = t == 0 ? (int)(y >> (6 * (TND - 1))) : (int)((y >> (6 * (TND - 1 - t))) & 63) - 32;
    const int block = g == 1 ? TND - 1 - t : t;
    *reinterpret_cast<__half*>(chunk + (uint32_t)block * kBlockB + ptx::sw_offset_b16<kRowB>((uint32_t)s, (uint32_t)q)) =
        __int2half_rn(digit);
  }
}

template <int GROUPS>
cudaError_t set_smem() {
  return cudaFuncSetAttribute(tri_kernel<GROUPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
}

}  // namespace

zp_status tri_launch(const TriArgs& a, int n_max, const int32_t* chunk_inst, int64_t n_chunks, bool gradients,
                     cudaStream_t stream) {
  if (a.n_items == 0 || n_chunks == 0) return ZP_OK;
  if (n_max > kTriMaxN) return set_error(ZP_ERR_INVALID_ARG, "triangle above its largest degree");
  static DeviceMemo<int> sms_memo;
  int sms = 0;
  ZP_TRY(sms_memo.get(&sms, [](int* x) -> zp_status {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(x, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = set_smem<1>();
    if (e == cudaSuccess) e = set_smem<2>();
    return e == cudaSuccess ? ZP_OK : cuda_error(e, "triangle kernel set-up");
  }));
  const int groups = gradients ? 2 : 1;
  int stages = kMaxBStages;
  while (smem_bytes(n_max, groups, stages) > kMaxSmem) --stages;
  // At least half of an SM's shared memory: one CTA per SM, since each takes all of tensor memory.
  const uint32_t smem = std::max<uint32_t>(smem_bytes(n_max, groups, stages), kMaxSmem / 2 + 4096);
  const unsigned grid = (unsigned)std::min<int64_t>(a.n_items, sms);
  if (gradients) tri_deriv_kernel<<<(unsigned)n_chunks, kTriChunk * TNS, 0, stream>>>(a, chunk_inst);
  tri_coeff_kernel<<<dim3((unsigned)n_chunks, (unsigned)groups), kTriChunk * TNS, 0, stream>>>(a, chunk_inst);
  if (gradients) tri_kernel<2><<<grid, kThreads, smem, stream>>>(a, n_max, stages);
  else tri_kernel<1><<<grid, kThreads, smem, stream>>>(a, n_max, stages);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ZP_OK : cuda_error(e, "triangle series launch");
}

TriInst tri_inst(const zp_plan* plan, const double* r, const double* theta, int64_t P, const double* coeffs, int64_t S) {
  TriInst d;
  d.n_max = plan->n_max;
  d.KC = tri_chunks(plan->n_max);
  d.seg_chunks = tri_segment_chunks(plan->n_max);
  d.J = plan->n_modes;
  d.P = P;
  d.S = S;
  d.r = r;
  d.theta = plan->tri_angles ? theta : nullptr;  // outputs without angles take any theta
  d.coeffs = coeffs;
  d.perm = plan->dev.tri_perm;
  return d;
}

static zp_status tri_single(TriArgs& a, const zp_plan* plan, bool gradients, cudaStream_t stream) {
  TriInst& d = a.single;
  const size_t digits = tri_digit_bytes(d.KC, gradients), cpos = gradients ? tri_cpos_bytes(d.KC) : 0;
  ScratchBuffer buf;
  ZP_TRY(buf.alloc(digits + cpos + 256, stream));
  d.bdig = (uint8_t*)buf.ptr;
  d.cpos = gradients ? (double*)((uint8_t*)buf.ptr + digits) : nullptr;
  d.cexp = (int*)((uint8_t*)buf.ptr + digits + cpos);
  a.n_items = (d.P + TM - 1) / TM;
  return tri_launch(a, plan->n_max, nullptr, d.KC, gradients, stream);
}

zp_status tri_series_eval(const zp_plan* plan, const double* r, const double* theta, int64_t P, const double* coeffs,
                          int64_t S, double* out, cudaStream_t stream) {
  TriArgs a;
  a.single = tri_inst(plan, r, theta, P, coeffs, S);
  a.single.out = out;
  return tri_single(a, plan, false, stream);
}

zp_status tri_point_grads(const zp_plan* plan, const double* r, const double* theta, int64_t P, const double* coeffs,
                          int64_t S, const double* G, double* grad_r, double* grad_theta, cudaStream_t stream) {
  if (P == 0 || (!grad_r && !grad_theta)) return ZP_OK;
  TriArgs a;
  a.single = tri_inst(plan, r, theta, P, coeffs, S);
  a.single.gdot = G;
  a.single.grad_r = grad_r;
  a.single.grad_theta = grad_theta;
  return tri_single(a, plan, true, stream);
}

zp_status tri_error_word(unsigned int* value, bool reset) {
  cudaError_t e = cudaMemcpyFromSymbol(value, g_tri_error, sizeof(unsigned int));
  if (e != cudaSuccess) return cuda_error(e, "cudaMemcpyFromSymbol");
  if (reset) {
    const unsigned int zero = 0;
    e = cudaMemcpyToSymbol(g_tri_error, &zero, sizeof(unsigned int));
    if (e != cudaSuccess) return cuda_error(e, "cudaMemcpyToSymbol");
  }
  return ZP_OK;
}

}  // namespace zp
