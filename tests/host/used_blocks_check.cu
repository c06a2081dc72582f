// Host check of the grid blocks a plan marks as used and of the spread lists
// cut down to them: every cell that a sample's footprint covers lies in a
// used block, every used block is covered by a footprint, and the lists
// write every cell of the used blocks once and no other cell.  Prints OK and
// exits 0 on success.
#include "plan.cu"
#include <cstdio>
#include <random>
using namespace prop;
int main() {
  int fails = 0;
  for (int W : {6, 8})
    for (int T : {1, 3})
      for (int n : {32, 48, 96, 1024}) {
        Plan p;
        p.n = n, p.N = n / 2, p.W = W, p.cs = 8, p.T = T, p.L = 2, p.R = 9;
        p.blade_frame = {0, T > 1 ? 2 : 0, 0};
        p.M = 3 * p.L * p.R;
        std::mt19937 rng(W + T + n);
        std::vector<int> tap(2 * p.M);
        for (int& v : tap) v = rng() % 2 ? (int)(rng() % n) : (n - 3 + (int)(rng() % 6)) % n;  // half of them at the seam
        std::vector<double> wd((size_t)p.M * 2 * W, 1.0);
        mark_used_blocks(p, tap);
        std::vector<char> want((size_t)T * n * n, 0), written(want.size(), 0), block(p.grid_used_h.size() * 64, 0);
        for (int m = 0; m < p.M; ++m)
          for (int a = 0; a < W; ++a)
            for (int b = 0; b < W; ++b) {
              const int t = p.blade_frame[m / (p.L * p.R)], r = (tap[2 * m + 1] + a) % n, c = (tap[2 * m] + b) % n;
              want[((size_t)t * n + r) * n + c] = 1;
              block[((size_t)t * (n / 2) + c / 2) * 64 + r / kGridBlock] = 1;
            }
        for (size_t i = 0; i < block.size(); ++i) fails += (p.grid_used_h[i / 64] >> (i % 64) & 1) != (uint64_t)block[i];
        std::vector<int4> items;
        std::vector<int2> blob;
        if (!build_group_lists(p, tap, wd, items, blob)) ++fails;
        for (const int4& it : items)
          for (int g = 0; g < it.y; ++g)
            for (int c = 0; c < 4; ++c) ++written[(size_t)blob[it.x + g].x + (size_t)(c >> 1) * n + (c & 1)];
        for (size_t i = 0; i < want.size(); ++i) {
          const size_t t = i / ((size_t)n * n), r = i / n % n, c = i % n;
          const int used = block[(t * (n / 2) + c / 2) * 64 + r / kGridBlock];
          fails += written[i] != used || want[i] > used;
        }
      }
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails != 0;
}
