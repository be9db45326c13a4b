// Host driver for tests/test_pair_walk.py: the triangle walk in pairs of float32 (zp_pair.h) at one point per
// line of stdin (hex floats), printing n, m and the float32 value of every radial polynomial.
//   argv[1] = n_max.  No GPU is touched.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "zp_pair.h"
#include "zp_tri.h"

using namespace zp;

int main(int, char** argv) {
  const int n_max = std::atoi(argv[1]), H = n_max / 2;
  char text[64];
  while (std::scanf("%63s", text) == 1) {
    const double rho = std::strtod(text, nullptr);
    const float rh = (float)rho, rl = (float)(rho - (double)rh);
    const float2 r = make_float2(rh, rl);
    std::vector<float2> st(2 * (n_max / 4) + 2);
    for (int A = 0; A <= H; ++A) {
      float2 l0 = make_float2(0.0f, 0.0f), l1 = l0, dg = make_float2(A == 0 ? -1.0f : 0.0f, 0.0f);
      for (int B = 0; B <= (A < H - A ? A : H - A); ++B) {
        const float2 u0 = B < A ? st[2 * B] : l0, u1 = B < A ? st[2 * B + 1] : l1;
        const float2 e00 = pair_step(r, u0, l0, dg), e01 = pair_step(r, u1, e00, u0);
        const float2 e10 = pair_step(r, e00, l1, l0), e11 = pair_step(r, e01, e10, e00);
        st[2 * B] = e10;
        st[2 * B + 1] = e11;
        dg = u1;
        l0 = e01;
        l1 = e11;
        const float2 e[4] = {e00, e01, e10, e11};
        for (int k = 0; k < 4; ++k) {
          const int a = 2 * A + (k >> 1), b = 2 * B + (k & 1);
          if (a + b <= n_max && a >= b) std::printf("%d %d %a\n", a + b, a - b, (double)e[k].x + (double)e[k].y);
        }
      }
    }
  }
  return 0;
}
