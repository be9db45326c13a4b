// Host driver for tests/test_tri_run.py: per degree the positions of a segment of the fused series'
// contraction, and the largest leading digit of a value digitised at its row's scale.  No GPU is touched.
#include <cstdio>
#include <cstdlib>

#include "zp_tri.h"

using namespace zp;

int main() {
  // A row's scale E has 2^E above 1.02 times its largest value: words y with |y| <= 2^62 / 1.02.
  const int64_t top = (int64_t)(0x1p62 / 1.02);
  const int hi = tri_digit((uint64_t)top + kTriWordBias, 0), lo = tri_digit((uint64_t)-top + kTriWordBias, 0);
  std::printf("%d %d\n", hi > -lo ? hi : -lo, kTriDigits);
  for (int n = 0; n <= kTriMaxN; ++n)
    std::printf("%d %d %d\n", tri_segment_chunks(n) * kTriChunk, tri_segments(n) * tri_segment_chunks(n), tri_chunks(n));
  return 0;
}
