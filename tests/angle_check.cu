// Host driver for tests/test_angles.py: per line of stdin (an angle as a hex float) whether the fixed-point
// table serves float64 results, then cos and sin of m theta at scale 2^62 for m = 1 .. argv[1].  No GPU is touched.
#include <cinttypes>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "zp_tri.h"

using namespace zp;

int main(int, char** argv) {
  char text[64];
  while (std::scanf("%63s", text) == 1) {
    const double th = std::strtod(text, nullptr);
    uint64_t bits;
    std::memcpy(&bits, &th, 8);
    int64_t ci, si;
    tri_cos_sin(tri_turn(bits), ci, si);
    std::printf("%d", tri_off_axes(ci, si, 53) ? 1 : 0);
    TriTrig c = tri_split(1ll << 62), s = tri_split(0);
    for (int m = 1; m <= std::atoi(argv[1]); ++m) {
      tri_rotate(c, s, tri_split(ci), tri_split(si));
      std::printf(" %" PRId64 " %" PRId64, (int64_t)c.hi * (1ll << 31) + c.lo, (int64_t)s.hi * (1ll << 31) + s.lo);
    }
    std::printf("\n");
  }
  return 0;
}
