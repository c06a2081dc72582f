// Host check of the shapes in which an update walks an image row (walk_shape):
// for every bin count and row length the blocks, groups and runs cover each
// (voxel, bin) of a row exactly once, no walk is longer than asked, and no more
// than a third of a block's threads is left over where the row is long enough.
// Prints OK and exits 0 on success.
#include "prop_internal.cuh"
#include <cstdio>
using namespace prop;

int main() {
  int fails = 0;
  for (int N : {8, 16, 24, 48, 96, 128, 192, 384, 512})
    for (int Nf = 1; Nf <= 700; Nf += Nf < 70 ? 1 : 23) {
      const int threads = 256, most = 8;
      const WalkShape w = walk_shape(Nf, N, threads, most);
      std::vector<int> seen((size_t)N * Nf, 0);
      bool ok = w.len >= 1 && w.len <= most && w.fw * w.runs <= threads && w.fw >= 1;
      for (int b = 0; b < w.nxb * w.nfg && ok; ++b)
        for (int tid = 0; tid < threads; ++tid) {
          const int run = tid / w.fw, f = b % w.nfg * w.fw + tid - run * w.fw;
          const int lo = (b / w.nfg * w.runs + run) * w.len, hi = std::min(N, lo + w.len);
          if (run >= w.runs || f >= Nf) continue;
          for (int i = lo; i < hi; ++i) ++seen[(size_t)i * Nf + f];
        }
      for (int v : seen) ok = ok && v == 1;
      if (3 * (long)w.fw * w.runs < 2 * threads && w.runs < N) ok = false;
      if (!ok && ++fails < 20) printf("N %d Nf %d: fw %d nfg %d runs %d len %d nxb %d\n", N, Nf, w.fw, w.nfg, w.runs, w.len, w.nxb);
    }
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails != 0;
}
