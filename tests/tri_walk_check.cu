// Host driver for tests/test_tri_walk.py: evaluates the fixed-point triangle walk (zp_tri.h) and
// prints the digits' values, and checks the contraction layout's two directions against each other.
//   argv[1] = n_max; stdin: lines "r theta" (hex floats).  No GPU is touched.
#include <cinttypes>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "zp_tri.h"

using namespace zp;

static uint64_t bits(double x) {
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return b;
}

int main(int, char** argv) {
  const int n_max = std::atoi(argv[1]), H = n_max / 2, positions = tri_chunks(n_max) * kTriChunk;
  std::vector<char> seen(positions, 0);
  for (int n = 0; n <= n_max; ++n)
    for (int m = n % 2; m <= n; m += 2)
      for (int h = 0; h < 2; ++h) {
        const int p = tri_position(n, m, h, n_max);
        int n2, m2, h2;
        tri_mode(p, n_max, n2, m2, h2);
        if (p < 0 || p >= positions || seen[p]++ || n2 != n || m2 != m || h2 != h) return 1;
      }
  if (tri_segment_chunks(n_max) * kTriChunk > kTriMaxRun) return 1;
  if (tri_segments(n_max) * tri_segment_chunks(n_max) < tri_chunks(n_max)) return 1;
  char a[64], b[64];
  while (std::scanf("%63s %63s", a, b) == 2) {
    const double r = std::strtod(a, nullptr), th = std::strtod(b, nullptr);
    const TriPoint tp = tri_point(bits(r));
    int64_t ci, si;
    tri_cos_sin(tri_turn(bits(th)), ci, si);
    std::vector<uint64_t> c, s, st(n_max + 4, kTriZero);
    TriTrig cm = tri_split(1ll << 62), sm = tri_split(0);
    for (int m = 0; m <= n_max + 1; ++m) {
      c.push_back(tri_entry(cm));
      s.push_back(tri_entry(sm));
      tri_rotate(cm, sm, tri_split(ci), tri_split(si));
    }
    std::vector<int64_t> out(positions, 0);
    int i = 0;
    for (int A = 0; A <= H; ++A) {
      uint64_t l0 = kTriZero, l1 = kTriZero, dg = A == 0 ? 0 : kTriZero;
      for (int B = 0; B <= (A < H - A ? A : H - A); ++B, ++i) {
        const uint64_t u0 = B < A ? st[2 * B] : l0, u1 = B < A ? st[2 * B + 1] : l1;
        const uint64_t e00 = tri_floor(tri_step(tp, u0, l0, dg)), e01 = tri_step(tp, u1, e00, u0);
        const uint64_t e10 = tri_step(tp, e00, l1, l0), e11 = tri_floor(tri_step(tp, e01, e10, e00));
        st[2 * B] = e10;
        st[2 * B + 1] = e11;
        dg = u1;
        l0 = e01;
        l1 = e11;
        const uint64_t e[4] = {e00, e01, e10, e11};
        const int m[4] = {2 * (A - B), 2 * (A - B) - 1, 2 * (A - B) + 1, 2 * (A - B)};
        for (int k = 0; k < 4; ++k)
          for (int h = 0; h < 2; ++h) {
            const uint64_t g = (h ? s : c)[m[k] < 0 ? 0 : m[k]];
            const uint64_t w = tri_word(e[k], g, tri_offset(g));
            int64_t x = 0;
            for (int t = 0; t < kTriDigits; ++t) x = x * 64 + tri_digit(w, t);
            out[i * 8 + h * 4 + k] = x;
          }
      }
    }
    for (int n = 0; n <= n_max; ++n)
      for (int m = n % 2; m <= n; m += 2)
        for (int h = 0; h < (m ? 2 : 1); ++h)
          std::printf("%d %d %" PRId64 "\n", n, h ? -m : m, out[tri_position(n, m, h, n_max)]);
  }
  return 0;
}
