// Host check of the interpolation's quads, without a GPU: for random blade
// angles (widths 6 and 8, every bin stride with quads, odd line and readout
// counts, frames, grid lengths down to 32 where a strip's window wraps) every
// sample is in exactly one quad; the window sums over a quad's record equal
// the sample's own W x W taps bit for bit; and a replay of the kernel's
// producer finds every row and column of every quad's window in its ring slot
// while the item may be read.  Prints OK and exits 0 on success.
#include "plan.cu"
#include <cstdio>
#include <random>
using namespace prop;
static int fails = 0;
#define CHECK(c) do { if (!(c)) { if (++fails < 20) printf("line %d: %s\n", __LINE__, #c); } } while (0)

template <int CS, int W>
void run(int n, int B, int L, int R, int T, int ctas) {
  using S = QuadShape<CS, W>;
  Plan p;
  p.n = n, p.N = n / 2, p.W = W, p.cs = CS, p.T = T, p.B = B, p.L = L, p.R = R, p.M = B * L * R;
  for (int b = 0; b < B; ++b) p.blade_frame.push_back(b * T / B);
  std::mt19937 rng(n + CS + W + L);
  std::uniform_real_distribution<double> angle(0, 3.14159265358979), weight(0.1, 1.0);
  std::vector<int> tap(2 * p.M);
  std::vector<double> wd((size_t)p.M * 2 * W);
  for (double& w : wd) w = weight(rng);
  for (int b = 0; b < B; ++b) {
    const double th = b == 0 ? 0.0 : b == 1 ? std::acos(-1.0) / 4 : angle(rng);
    for (int l = 0; l < L; ++l)
      for (int j = 0; j < R; ++j) {
        const double kp = (l - L / 2.0) / p.N, kr = (j - R / 2.0) / p.N;
        const double k[2] = {kr * std::cos(th) - kp * std::sin(th), kr * std::sin(th) + kp * std::cos(th)};
        for (int a = 0; a < 2; ++a) {
          double u = n * k[a];
          u -= n * std::floor(u / n);
          tap[2 * ((b * L + l) * R + j) + a] = ((int)std::floor(u) - (W / 2 - 1) + n) % n;
        }
      }
  }
  std::vector<float4> quads;
  std::vector<int4> items;
  std::vector<int> off;
  build_quads(p, tap, wd, ctas, quads, items, off);
  CHECK((int)off.size() - 1 <= ctas && off[0] == 0 && off.back() == (int)items.size());
  std::vector<float> grid((size_t)T * n * n);
  for (float& g : grid) g = (float)weight(rng) - 0.5f;
  std::vector<int> seen(p.M, 0);
  const int TC = quad_cols(CS), nstrip = (n + TC - 1) / TC;
  int nq = 0;
  for (size_t c = 0; c + 1 < off.size(); ++c) {
    CHECK(off[c] < off[c + 1]);
    // the producer's schedule
    std::vector<long> row_in(S::NR, -1);  // (strip, row) in each slot
    std::vector<int> first_of;
    int released = 0, loaded = 0, first = 0, strip = -1, row = 0, row_end = 0;
    for (int k = 0; off[c] + k < off[c + 1]; ++k) {
      const int4 it = items[off[c] + k];
      CHECK(it.y == nq && it.z >= 1 && it.z <= S::ITEM);
      nq += it.z;
      const int st = it.x, r0 = it.w & 0xffff, nr = it.w >> 16;
      CHECK(r0 < n && nr >= W && nr <= S::SPAN - 1 + S::UW);
      released = std::max(released, k - kQuadStages + 1);
      int fresh = 0;
      if (st == strip && r0 < row_end) {
        CHECK(r0 >= row);
        first += r0 - row;
        fresh = std::min(nr, row_end - r0);
      } else {
        first = loaded;
      }
      first_of.push_back(first);
      for (int i = fresh; i < nr; ++i) {
        while (released < k && first_of[released] + S::NR <= first + i) ++released;
        row_in[(first + i) % S::NR] = (long)st * n + (r0 + i) % n;
      }
      loaded = std::max(loaded, first + nr);
      strip = st, row = r0;
      row_end = std::max(fresh > 0 ? row_end : 0, r0 + nr);
      const int t = st / nstrip, c0 = (st - t * nstrip) * TC;
      const int cells = std::min(S::HC, n - c0 + S::UW - 1);
      CHECK(cells - std::min(cells, n - c0) <= n);
      // every item that may be read now has its rows
      for (int j = released; j <= k; ++j) {
        const int4 ij = items[off[c] + j];
        for (int i = 0; i < (ij.w >> 16); ++i)
          CHECK(row_in[(first_of[j] + i) % S::NR] == (long)ij.x * n + ((ij.w & 0xffff) + i) % n);
      }
      for (int q = 0; q < it.z; ++q) {
        const float* w = reinterpret_cast<const float*>(&quads[(size_t)(it.y + q) * S::REC]);
        const int* tail = reinterpret_cast<const int*>(w + 8 * S::UW);
        const int rows = tail[7] & 0xff, cols = tail[7] >> 8;
        CHECK(rows <= S::UW && cols >= W && cols <= S::UW && tail[4] + rows <= nr && tail[5] + S::UW <= S::HC);
        CHECK(tail[5] + cols <= cells && tail[6] >= 0 && tail[6] < R && (tail[1] < 0 || tail[6] + 1 < R));
        for (int s = 0; s < 4; ++s) {
          const int m = tail[s];
          if (m < 0) continue;
          CHECK(m < p.M && m % R == tail[6] + s % 2 && p.blade_frame[m / (L * R)] == t);
          ++seen[m];
          float got = 0.f, want = 0.f;
          for (int r = 0; r < rows; ++r) {
            float rs = 0.f;
            for (int x = 0; x < cols; ++x)
              rs = fmaf(w[4 * x + s], grid[((size_t)t * n + (r0 + tail[4] + r) % n) * n + (c0 + tail[5] + x) % n], rs);
            got = fmaf(w[4 * (S::UW + r) + s], rs, got);
          }
          for (int r = 0; r < W; ++r) {
            float rs = 0.f;
            for (int x = 0; x < W; ++x)
              rs = fmaf((float)wd[(size_t)m * 2 * W + x],
                        grid[((size_t)t * n + (tap[2 * m + 1] + r) % n) * n + (tap[2 * m] + x) % n], rs);
            want = fmaf((float)wd[(size_t)m * 2 * W + W + r], rs, want);
          }
          CHECK(got == want);
        }
      }
    }
  }
  for (int m = 0; m < p.M; ++m) CHECK(seen[m] == 1);
}

template <int CS>
void widths(int n, int B, int L, int R, int T, int ctas) {
  run<CS, 6>(n, B, L, R, T, ctas);
  run<CS, 8>(n, B, L, R, T, ctas);
}

int main() {
  const int g[][6] = {{32, 3, 4, 16, 1, 5},   {32, 1, 1, 1, 1, 152}, {48, 5, 3, 25, 2, 7},  {96, 7, 5, 53, 3, 152},
                      {128, 4, 33, 70, 4, 9}, {512, 3, 9, 256, 1, 152}, {64, 40, 16, 64, 1, 3}};
  for (auto& q : g) {
    widths<8>(q[0], q[1], q[2], q[3], q[4], q[5]);
    widths<16>(q[0], q[1], q[2], q[3], q[4], q[5]);
    widths<32>(q[0], q[1], q[2], q[3], q[4], q[5]);
    widths<64>(q[0], q[1], q[2], q[3], q[4], q[5]);
  }
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails != 0;
}
