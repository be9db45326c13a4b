// Host driver for tests/test_tri_index.py: runs the triangle kernels' block order over every chunk of every
// degree, the padding block included, against the sizes of what they index.  No GPU is touched.
#include <cstdio>

#include "zp_tri.h"

using namespace zp;

int main() {
  for (int n_max = 0; n_max <= kTriMaxWalkN; ++n_max) {
    const int H = n_max / 2, rows = tri_state_rows(n_max), blocks = tri_blocks(n_max);
    TriBlock bi;  // the fused series: two blocks per chunk
    for (int i = 0; i < 2 * tri_chunks(n_max); ++i, bi.advance(H)) {
      if (bi.B < 0 || 2 * bi.B + 1 >= rows) return std::printf("state row %d %d\n", n_max, i), 1;
      if (i < blocks && (bi.A != tri_row_of(i, H) || bi.B != i - tri_blocks_before(bi.A, H)))
        return std::printf("order %d %d\n", n_max, i), 1;
      const int m0 = 2 * (bi.A - bi.B);
      const TriAngleRows am = tri_angle_rows(m0, n_max);
      const int found[3] = {am.low, am.mid, am.top};
      for (int d = -1; d <= 1; ++d) {
        const int m = m0 + d, row = found[d + 1];
        if (m0 < 0 || row < 0 || row > n_max) return std::printf("angle row %d %d\n", n_max, i), 1;
        if (i < blocks && m >= 0 && m <= n_max && row != m) return std::printf("angle %d %d\n", n_max, i), 1;
      }
      // A block reads the row above where the one before it has been written.
      if (i < blocks && bi.B < bi.A && bi.B > (bi.A - 1 < H - (bi.A - 1) ? bi.A - 1 : H - (bi.A - 1)))
        return std::printf("row above %d %d\n", n_max, i), 1;
    }
    int i = 0;  // the other walks: two nested loops
    for (int A = 0; A <= H; ++A)
      for (int B = 0; B <= (A < H - A ? A : H - A); ++B, ++i)
        if (2 * B + 1 >= rows || 2 * (A + B) + 2 > n_max + 2 || i >= blocks) return std::printf("loops %d %d\n", n_max, i), 1;
    if (i != blocks) return std::printf("blocks %d\n", n_max), 1;
  }
  return 0;
}
