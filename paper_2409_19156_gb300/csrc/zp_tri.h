// Fixed-point evaluation of every Zernike function of a triangle n <= n_max at one point, on the
// integer pipe, and the contraction layout that goes with it (zp_tri.cu).
//
// GB300 issues a float64 operation on two lanes per SM and clock and a 32 x 32 -> 64 bit integer
// multiply-add on at least sixteen times as many, so on the unit disc, where every |R_n^m| <= 1,
// 64-bit fixed point is both faster and more accurate than float64.  The recursion in n for each
// m amplifies absolute errors while R_n^m grows from rho^m, so fixed point takes the recursion
// over neighbouring m instead (R_n^m = rho (R_{n-1}^{|m-1|} + R_{n-1}^{m+1}) - R_{n-2}^m, from
// R_n^m = (1 / 2 pi) int U_n(rho cos t) cos(m t) dt and U_n = 2x U_{n-1} - U_{n-2}): it has no
// growing solution (an error made at one (n, m) spreads as the radial functions themselves, at
// most 1 in magnitude), no tables, and one multiplication per value.
//
// With a = (n + |m|) / 2 and b = (n - |m|) / 2 (the Jacobi degree) it reads
//   f(a, b) = rho (f(a-1, b) + f(a, b-1)) - f(a-1, b-1),   f(a, b) = f(b, a),   f(0, 0) = 1,
// walked in 2 x 2 blocks (a = 2A, 2A+1; b = 2B, 2B+1), A ascending and B = 0 .. min(A, H - A)
// with H = n_max / 2: one stored row f(2A-1, .) of at most H + 2 values is the whole state.
// The elements of a block are e00 = f(2A, 2B), e01 = f(2A, 2B+1), e10 = f(2A+1, 2B) and
// e11 = f(2A+1, 2B+1), of |m| = 2(A-B), 2(A-B)-1, 2(A-B)+1 and 2(A-B).  e01 of a diagonal block
// (m = -1) and elements above n_max hold no mode.
//
// Contraction layout: chunk k of 16 positions holds blocks 2k and 2k+1, each the cos values of its
// four elements, then their sin values.
#pragma once

#include <cstdint>

namespace zp {

constexpr int kTriMaxN = 64;      // largest n_max (shared memory for a tile's state and angles)
constexpr int kTriMaxWalkN = 256; // largest n_max of the float64 walk over the same layout
constexpr int kTriDigits = 9;     // base-64 digits per value
constexpr int kTriChunk = 16;     // positions per chunk (one tensor-core K step)
// Longest run of positions whose diagonal sums stay below 2^24 (exact in float32): digits of at
// most 63 (values; 33 on the disc, but a row off it is scaled to just below twice that) and 65
// (coefficients) in front, 32 behind, so a position adds at most 63 * 32 + 65 * 32 + 7 * 32^2 = 11264 to
// the largest kept diagonal.
constexpr int kTriMaxRun = 1489;  // positions: 1489 * 11264 < 2^24

// The number of blocks in rows before A, and in all rows, of the triangle with H = n_max / 2.
__host__ __device__ constexpr int tri_blocks_before(int A, int H) {
  // Rows A' hold min(A', H - A') + 1 blocks: ascending up to A' = H / 2, then descending.
  const int h = H / 2;
  if (A <= h + 1) return A * (A + 1) / 2;
  const int r = H - A + 1;  // blocks of row A (and r, r - 1, .., 1 still to come)
  const int up = (h + 1) * (h + 2) / 2;
  const int down_all = (H - h) * (H - h + 1) / 2;  // rows h+1 .. H hold H-h, .., 1 blocks
  return up + down_all - r * (r + 1) / 2;
}
__host__ __device__ constexpr int tri_blocks(int n_max) { return tri_blocks_before(n_max / 2 + 1, n_max / 2); }
__host__ __device__ constexpr int tri_chunks(int n_max) { return (tri_blocks(n_max) + 1) / 2; }
// Segments of a contraction (each with its own accumulator) and chunks per segment.
__host__ __device__ constexpr int tri_segments(int n_max) {
  return (tri_chunks(n_max) * kTriChunk + kTriMaxRun - 1) / kTriMaxRun;
}
__host__ __device__ constexpr int tri_segment_chunks(int n_max) {
  return (tri_chunks(n_max) + tri_segments(n_max) - 1) / tri_segments(n_max);
}
// Position of mode (n, |m|), sine or cosine, in the contraction.
__host__ __device__ constexpr int tri_position(int n, int am, int sine, int n_max) {
  const int a = (n + am) / 2, b = (n - am) / 2;
  const int i = tri_blocks_before(a / 2, n_max / 2) + b / 2;
  return i * 8 + sine * 4 + (a & 1) * 2 + (b & 1);
}
// The block row A that holds block i.
__host__ __device__ constexpr int tri_row_of(int i, int H) {
  int A = 0;
  while (A < H && tri_blocks_before(A + 1, H) <= i) ++A;
  return A;
}
// Mode at position p: n and |m| (m = -1 marks the unused element of a diagonal block).
__host__ __device__ constexpr void tri_mode(int p, int n_max, int& n, int& m, int& sine) {
  const int H = n_max / 2;
  const int i = p / 8;
  const int A = tri_row_of(i, H), B = i - tri_blocks_before(A, H);
  const int a = 2 * A + ((p >> 1) & 1), b = 2 * B + (p & 1);
  n = i < tri_blocks(n_max) ? a + b : n_max + 1;
  m = a - b;
  sine = (p >> 2) & 1;
}

// The order of a point's blocks: row A, block B of 0 .. nb.  An odd number of blocks leaves the last chunk
// one more, past the last row (B = 0): its values have no modes.
struct TriBlock {
  int A = 0, B = 0, nb = 0;
  __host__ __device__ __forceinline__ void advance(int H) {
    const bool end = B == nb;
    A += end;
    B = end ? 0 : B + 1;
    nb = A < H - A ? A : H - A;
  }
};
// Rows of the stored row above (two per block).
__host__ __device__ constexpr int tri_state_rows(int n_max) { return 2 * (n_max / 4) + 2; }
// Rows of an angle table [0, n_max] for a block of |m| = m0 - 1 (e01), m0 (e00, e11) and m0 + 1 (e10), m0 >= 0;
// elements without a mode take a row that exists.
struct TriAngleRows {
  int low, mid, top;
};
__host__ __device__ __forceinline__ TriAngleRows tri_angle_rows(int m0, int n_max) {
  const int low = m0 > 0 ? m0 - 1 : 0;
  return {low < n_max ? low : n_max, m0 < n_max ? m0 : n_max, m0 + 1 < n_max ? m0 + 1 : n_max};
}

// ------------------------------------------------------------------ arithmetic (host and device)

__host__ __device__ __forceinline__ uint64_t tri_umul_hi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// Biased state: f in [-1, 1] as (f + 1) 2^61.
constexpr uint64_t kTriZero = 1ull << 61;

struct TriPoint {
  uint64_t rho;   // rho 2^64 (rho = 1: 2^64 - 1)
  uint64_t bias;  // (2 - 2 rho) 2^61, plus one unit against the truncations of tri_mul_add
};

// rho in [0, 1] of a float64, by its bits.
__host__ __device__ __forceinline__ TriPoint tri_point(uint64_t rho_bits) {
  const int e = (int)((rho_bits >> 52) & 0x7ffu);  // the sign can only be -0's
  const uint64_t mant = (rho_bits & 0xfffffffffffffull) | (1ull << 52);
  TriPoint t;
  if (e >= 1023) {
    t.rho = ~0ull;
  } else {
    const int sh = e - 1023 - 52 + 64;  // rho 2^64 = mant 2^sh
    t.rho = e == 0 ? 0 : (sh >= 0 ? mant << sh : (sh > -64 ? mant >> -sh : 0));
  }
  t.bias = (1ull << 62) - (t.rho >> 2) + 1;
  return t;
}

// High word of s g plus `add`, from three of the four 32-bit partial products (the lowest one and
// two low-word carries dropped, 1.25 units on average).  Unsigned on purpose: the signed 32 x 32
// -> 64 bit multiply takes several instructions on sm_103a, the unsigned one is a single one; and
// the device form spells the carries out (8 instructions after the sums, against 11 from C).
__host__ __device__ __forceinline__ uint64_t tri_mul_add(uint64_t s, uint64_t g, uint64_t add) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("{\n\t.reg .u32 sl, sh, gl, gh, x, y, rl, rh;\n\t.reg .u64 q;\n\t"
      "mov.b64 {sl, sh}, %1;\n\tmov.b64 {gl, gh}, %2;\n\t"
      "mul.hi.u32 x, sl, gh;\n\tmul.hi.u32 y, sh, gl;\n\t"
      "mad.wide.u32 q, sh, gh, %3;\n\tmov.b64 {rl, rh}, q;\n\t"
      "add.cc.u32 rl, rl, x;\n\taddc.u32 rh, rh, 0;\n\t"
      "add.cc.u32 rl, rl, y;\n\taddc.u32 rh, rh, 0;\n\t"
      "mov.b64 %0, {rl, rh};\n\t}"
      : "=l"(r)
      : "l"(s), "l"(g), "l"(add));
  return r;
#else
  const uint32_t sl = (uint32_t)s, sh = (uint32_t)(s >> 32), gl = (uint32_t)g, gh = (uint32_t)(g >> 32);
  return (uint64_t)sh * gh + add + (((uint64_t)sl * gh) >> 32) + (((uint64_t)sh * gl) >> 32);
#endif
}

// rho (f1 + f2) - f0 on biased words.
__host__ __device__ __forceinline__ uint64_t tri_step(const TriPoint& t, uint64_t f1, uint64_t f2, uint64_t f0) {
  return tri_mul_add(f1 + f2, t.rho, t.bias - f0);
}

// A biased word kept from wrapping below -1: R_n^0 comes that close near the origin (n = 2 mod 4), and
// tri_word takes the word as unsigned.  Only m = 0 needs it: elements e00 and e11.
__host__ __device__ __forceinline__ uint64_t tri_floor(uint64_t f) { return (int64_t)f < 0 ? 0 : f; }

// A signed number of [-1, 1] at scale 2^62 as a high word (31 bits down) and 31 low bits.
struct TriTrig {
  int32_t hi;
  uint32_t lo;
};
__host__ __device__ __forceinline__ TriTrig tri_split(int64_t v) {
  // Rounding may carry a cosine of +-1 just beyond the range.
  const int64_t top = (1ll << 62) - 1, bottom = -(1ll << 62);
  v = v > top ? top : (v < bottom ? bottom : v);
  TriTrig t;
  t.hi = (int32_t)(v >> 31);
  t.lo = (uint32_t)v & 0x7fffffffu;
  return t;
}

// Offset of a digitised word: 2^62 makes the leading digit positive, 32 at each later digit
// balances it, half a unit of the last digit rounds.
constexpr uint64_t tri_word_bias() {
  uint64_t b = (1ull << 62) + (1ull << 7);
  for (int k = 0; k < kTriDigits - 1; ++k) b += 32ull << (8 + 6 * k);
  return b;
}
constexpr uint64_t kTriWordBias = tri_word_bias();

// An angle table's entry: (trig + 1) / 2 at scale 2^64.
__host__ __device__ __forceinline__ uint64_t tri_entry(const TriTrig& t) {
  const int64_t v = (int64_t)t.hi * (1ll << 31) + t.lo;
  return ((uint64_t)v + (1ull << 62)) << 1;
}
// kTriWordBias - trig 2^61 of an entry.
__host__ __device__ __forceinline__ uint64_t tri_offset(uint64_t entry) {
  return kTriWordBias + (1ull << 61) - (entry >> 2);
}
// f trig as a word y 2^61 + kTriWordBias: with f' = f + 1 (biased) and g = (trig + 1) / 2,
// f trig = 2 f' g - f' - trig.
__host__ __device__ __forceinline__ uint64_t tri_word(uint64_t f, uint64_t entry, uint64_t offset) {
  return tri_mul_add(f + f, entry, offset - f);
}

// Digit d of a word as an integer: the leading one in [-64, 64), later ones in [-32, 32).
__host__ __device__ __forceinline__ int tri_digit(uint64_t w, int d) {
  return d == 0 ? (int)((w >> 56) & 127u) - 64 : (int)((w >> (56 - 6 * d)) & 63u) - 32;
}

// a b for two split numbers, at scale 2^62 (truncated, below one unit).
__host__ __device__ __forceinline__ int64_t tri_mul(const TriTrig& a, const TriTrig& b) {
  const int64_t mid = (int64_t)a.hi * (int32_t)b.lo + (int64_t)(int32_t)a.lo * b.hi;
  return (int64_t)a.hi * b.hi + (mid >> 31);
}

// A float64 angle, |theta| < 2^52, as a fraction of a turn at scale 2^64 (whole turns dropped):
// theta times 128 bits of 1 / (2 pi), within 1.5 units.  Multiples of the angle are multiples of the word.
constexpr int kTriAngleExponent = 1023 + 52;  // biased exponents below it
__host__ __device__ __forceinline__ uint64_t tri_turn(uint64_t theta_bits) {
  const int e = (int)((theta_bits >> 52) & 0x7ffu);
  const uint64_t mant = e ? (theta_bits & 0xfffffffffffffull) | (1ull << 52) : 0ull;
  // floor(2^128 / (2 pi)), high and low words.
  constexpr uint64_t kI1 = 0x28be60db9391054aull, kI0 = 0x7f09d5f47d4d3770ull;
  const uint64_t p0 = mant * kI1, q0 = tri_umul_hi(mant, kI0);
  const uint64_t ql = p0 + q0, qh = tri_umul_hi(mant, kI1) + (ql < p0 ? 1u : 0u);
  const int sh = 1075 - e;  // turn = (qh 2^64 + ql) 2^-sh mod 2^64; sh >= 1
  const uint64_t turn = sh < 64 ? (qh << (64 - sh)) | (ql >> sh) : (sh < 128 ? qh >> (sh - 64) : 0ull);
  return theta_bits >> 63 ? 0 - turn : turn;
}

// cos and sin of a fraction of a turn, at scale 2^62: the nearest quarter turn taken off, Taylor's
// series of the rest (|x| <= pi / 4) in 64-bit fixed point.
__host__ __device__ __forceinline__ void tri_cos_sin(uint64_t turn, int64_t& c, int64_t& s) {
  const uint32_t k = (uint32_t)((turn + (1ull << 61)) >> 62);
  const int64_t r = (int64_t)(turn - ((uint64_t)k << 62));
  uint64_t ar = r < 0 ? (uint64_t)(-r) : (uint64_t)r;
  if (ar >> 61) ar = (1ull << 61) - 1;
  const uint64_t x = tri_umul_hi(ar << 3, 0xc90fdaa22168c234ull);  // |x| 2^64 (times pi / 4)
  const uint64_t u = tri_umul_hi(x, x);
  uint64_t hc = 0x8ull, hs = 0x98ull;
  // 2^64 / (2 i)! and 2^64 / (2 i + 1)!, innermost first.
  hc = 0xb41ull - tri_umul_hi(u, hc);
  hc = 0xd73faull - tri_umul_hi(u, hc);
  hs = 0xca96ull - tri_umul_hi(u, hs);
  hc = 0xc9cba54ull - tri_umul_hi(u, hc);
  hs = 0xd73f9full - tri_umul_hi(u, hs);
  hc = 0x8f76c77fcull - tri_umul_hi(u, hc);
  hs = 0xb092309dull - tri_umul_hi(u, hs);
  hc = 0x49f93edde28ull - tri_umul_hi(u, hc);
  hs = 0x6b99159fd5ull - tri_umul_hi(u, hs);
  hc = 0x1a01a01a01a02ull - tri_umul_hi(u, hc);
  hs = 0x2e3bc74aad8eull - tri_umul_hi(u, hs);
  hc = 0x5b05b05b05b05bull - tri_umul_hi(u, hc);
  hs = 0xd00d00d00d00dull - tri_umul_hi(u, hs);
  hc = 0xaaaaaaaaaaaaaabull - tri_umul_hi(u, hc);
  hs = 0x222222222222222ull - tri_umul_hi(u, hs);
  hc = 0x8000000000000000ull - tri_umul_hi(u, hc);
  hs = 0x2aaaaaaaaaaaaaabull - tri_umul_hi(u, hs);
  const int64_t cq = (int64_t)((1ull << 62) - (tri_umul_hi(u, hc) >> 2));
  const uint64_t w = tri_umul_hi(u, hs);
  const uint64_t g = w ? 0 - w : ~0ull;
  int64_t sq = (int64_t)(tri_umul_hi(x, g) >> 2);
  if (r < 0) sq = -sq;
  c = (k & 1) ? ((k & 2) ? sq : -sq) : ((k & 2) ? -cq : cq);
  s = (k & 1) ? ((k & 2) ? -cq : cq) : ((k & 2) ? -sq : sq);
}

// Whether cos and sin of an angle (scale 2^62) both leave `bits` bits of themselves in fixed point: next to a
// multiple of a quarter turn one of them, and the like multiples' with it, is too small.
__host__ __device__ __forceinline__ bool tri_off_axes(int64_t c, int64_t s, int bits) {
  const int64_t ac = c < 0 ? -c : c, as = s < 0 ? -s : s;
  return ((ac < as ? ac : as) >> bits) != 0;
}

// The next angle of a table: (c, s) turned by (c1, s1).  The m-th is within (m + 1) 10 2^-62: of that up to 2.4
// per m from the word of the turn, 4 of the first angle's own, and two truncated products.
__host__ __device__ __forceinline__ void tri_rotate(TriTrig& c, TriTrig& s, const TriTrig& c1, const TriTrig& s1) {
  const int64_t cn = tri_mul(c, c1) - tri_mul(s, s1);
  const int64_t sn = tri_mul(s, c1) + tri_mul(c, s1) + 1;
  c = tri_split(cn);
  s = tri_split(sn);
}

}  // namespace zp
