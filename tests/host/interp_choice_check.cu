// Host check, without a GPU, of the interpolation tiles and of the rule that
// takes tiles or quads.  Tiles: every sample is in exactly one item, with its
// first tap in the item's tile, an item has at most kInterpItem samples, and the
// CTAs' ranges cover the items.  The rule, on a device of 152 SMs: geometries
// that measured clearly faster one way or the other.  Prints OK and exits 0 on
// success.
#include "plan.cu"
#include <cstdio>
using namespace prop;
static int fails = 0;
#define CHECK(c) do { if (!(c)) { if (++fails < 20) printf("line %d: %s\n", __LINE__, #c); } } while (0)

static bool takes_quads(int N, int Nf, int B, int L, int R, int T, int W) {
  Plan p;
  p.N = N, p.n = 2 * N, p.W = W, p.cs = Nf + (Nf & 1), p.T = T, p.B = B, p.L = L, p.R = R, p.M = B * L * R;
  std::vector<int> tap;
  const double pi = std::acos(-1.0), golden = pi * (std::sqrt(5.0) - 1) / 2;
  for (int b = 0; b < B; ++b) {
    p.blade_frame.push_back(b * T / B);
    const double th = T == 1 ? pi * b / B : std::fmod(b * golden, pi);
    for (int l = 0; l < L; ++l)
      for (int j = 0; j < R; ++j) {
        const double kp = (l - L / 2.0) / N, kr = (j - R / 2.0) / N;
        const double k[2] = {kr * std::cos(th) - kp * std::sin(th), kr * std::sin(th) + kp * std::cos(th)};
        for (int a = 0; a < 2; ++a) {
          double u = p.n * k[a];
          u -= p.n * std::floor(u / p.n);
          tap.push_back(((int)std::floor(u) - (W / 2 - 1) + p.n) % p.n);
        }
      }
  }
  std::vector<int> order, off, qoff;
  std::vector<int4> items, qitems;
  std::vector<float4> quads;
  build_tiles(p, tap, 152, order, items, off);
  const int TR = interp_tile_rows(p.cs, W), TC = interp_tile_cols(p.cs);
  const int nct = p.n / TC, tpf = (p.n + TR - 1) / TR * nct;
  std::vector<int> seen(p.M, 0);
  CHECK((int)off.size() - 1 <= 152 && off[0] == 0 && off.back() == (int)items.size());
  for (size_t c = 0; c + 1 < off.size(); ++c) CHECK(off[c] < off[c + 1]);
  for (const int4& it : items) {
    CHECK(it.z >= 1 && it.z <= kInterpItem);
    const int t = it.x / tpf, r0 = it.x % tpf / nct * TR, c0 = it.x % nct * TC;
    for (int i = it.y; i < it.y + it.z; ++i) {
      const int m = order[i];
      ++seen[m];
      CHECK(p.blade_frame[m / (L * R)] == t);
      CHECK(tap[2 * m] >= c0 && tap[2 * m] < c0 + TC && tap[2 * m + 1] >= r0 && tap[2 * m + 1] < r0 + TR);
    }
  }
  for (int m = 0; m < p.M; ++m) CHECK(seen[m] == 1);
  if (!quad_stride(p.cs)) return false;
  const std::vector<double> wd((size_t)p.M * 2 * W, 1.0);
  mark_used_blocks(p, tap);
  build_quads(p, tap, wd, 152, quads, qitems, qoff);
  return quads_time(p, qitems, qoff).longest < tiles_time(p, items, off).longest;
}

int main() {
  // quads: dense samples, or many in few tiles
  CHECK(takes_quads(256, 32, 16, 24, 256, 1, 8));
  CHECK(takes_quads(192, 16, 64, 16, 192, 32, 8));
  CHECK(takes_quads(512, 16, 12, 32, 512, 1, 6));
  CHECK(takes_quads(32, 64, 48, 4, 32, 1, 8));
  CHECK(takes_quads(16, 8, 16, 32, 16, 1, 8));
  CHECK(takes_quads(128, 8, 64, 16, 128, 32, 8));
  CHECK(takes_quads(64, 31, 48, 8, 64, 1, 8));
  // tiles: few samples a frame, one line a blade, 64 bins at width 8
  CHECK(!takes_quads(16, 64, 64, 4, 16, 32, 8));
  CHECK(!takes_quads(192, 64, 64, 1, 192, 32, 8));
  CHECK(!takes_quads(192, 64, 64, 16, 192, 32, 8));
  CHECK(!takes_quads(256, 64, 16, 24, 256, 1, 8));
  CHECK(!takes_quads(32, 63, 8, 32, 32, 8, 8));
  CHECK(!takes_quads(64, 32, 8, 8, 64, 8, 6));
  // other strides: tiles of their own sizes
  CHECK(!takes_quads(48, 5, 7, 11, 49, 3, 8));
  CHECK(!takes_quads(24, 40, 3, 5, 25, 2, 6));
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails != 0;
}
