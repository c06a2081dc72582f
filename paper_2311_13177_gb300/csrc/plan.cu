// Plan builder: validates the geometry, computes every table in FP64 on the
// host, stores them in FP32 on the device, and sizes the workspace.
//
// Tables (all from the operator y_b(k) = s sum_f P sum_x V exp(-2 pi i k.x)
// evaluated by a Kaiser-Bessel NUFFT with oversampling 2 and width 6):
//   * per sample m = (b L + l) R + j: k = k_r d_b + k_p d_b^perp, grid
//     coordinate u = 2N k (mod 2N, exact because the sum over integer x is
//     1-periodic in k), first tap floor(u) - (W/2 - 1) and the W weights per
//     axis psi(u - tap), psi(t) = I0(beta sqrt(1 - (2t/W)^2)) / I0(beta);
//   * deapodisation c(x) = I0(beta) / psihat(x / 2N) with the closed-form
//     transform psihat(xi) = W sinh(sqrt(beta^2 - (pi W xi)^2)) / sqrt(...),
//     beta = pi sqrt((W/sigma)^2 (sigma - 1/2)^2 - 0.8) (Beatty et al. 2005);
//   * displacement phase P[j][f] = exp(-2 pi i k_r Delta_f), the argument
//     k_r Delta_f reduced modulo 1 in FP64 before the cosine and sine
//     (Sec. 3: a displacement along the readout is a phase linear in k_r);
//   * FFT twiddles exp(-2 pi i q / 2N);
//   * interpolation order (samples sorted by grid tile) and spread gather
//     lists: for every grid cell the (sample, weight) pairs that cover it.
#include "prop_internal.cuh"

#include <cmath>
#include <cstring>
#include <algorithm>
#include <new>

namespace prop {

namespace {

// Modified Bessel function of the first kind, order 0, from its power series
// I0(z) = sum_k ((z/2)^(2k)) / (k!)^2 (all terms positive, so the partial sums
// converge monotonically; 60 terms reach double precision for z <= 40).
double bessel_i0(double z) {
  const double q = 0.25 * z * z;
  double term = 1.0, sum = 1.0;
  for (int k = 1; k < 60; ++k) {
    term *= q / ((double)k * (double)k);
    sum += term;
    if (term < 1e-17 * sum) break;
  }
  return sum;
}

bool fft_size_supported(int n) {
  static const int ok[] = {16, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024};
  for (int v : ok)
    if (v == n) return true;
  return false;
}

// Grouped spread lists for the shared-memory staged spread kernel.  The
// grid cells of every frame are cut into 2 x 2-cell groups; a group's list
// holds every sample whose W x W footprint meets the group, in ascending m,
// as (phased-residual offset m * cs, the sample's weight w2[a] w1[b] on each
// of the group's four cells, row-major, zero where the footprint misses the
// cell).  The weights are the FP64 products rounded once, as in the
// interpolation's tables, so every cell accumulates the same terms in the
// same order as a per-cell list would.  Every list is padded to a multiple
// of four entries with (row M, zero weights), row M of the phased residual
// being kept zero.  Groups are taken in frame, 4 x 4-group patch, row-major
// order, those in grid blocks that no sample reaches (grid_used_h) left out,
// and cut into items of about equal work, each item one blob of int2
// words staged by a single bulk copy:
//   groups[ngp]      (first cell index, end of its list), ngp = ngroups rounded up to even
//   offs[nent / 2]   nent int32 offsets (nent a multiple of 4)
//   wts[2 nent]      nent float4 weights
// Returns false when one group's list alone exceeds a stage.
bool build_group_lists(const Plan& p, const std::vector<int>& first_tap, const std::vector<double>& wd,
                       std::vector<int4>& sitems, std::vector<int2>& blob) {
  const int n = p.n, W = p.W, G = kSpreadGroup, gps = n / G, PG = kSpreadGroupPatch;
  static_assert(kSpreadGroup == 2, "four weights per entry");
  const size_t LR = (size_t)p.L * p.R;
  const size_t ngroup = (size_t)p.T * gps * gps;
  auto axis_groups = [&](int first, int* out) {
    int cnt = 0;
    for (int a = 0; a < W; ++a) {
      const int g = ((first + a) % n) / G;
      bool seen = false;
      for (int k = 0; k < cnt; ++k) seen = seen || out[k] == g;
      if (!seen) out[cnt++] = g;
    }
    return cnt;
  };
  std::vector<int> gcnt(ngroup, 0);
  for (size_t m = 0; m < (size_t)p.M; ++m) {
    const size_t frame = (size_t)p.blade_frame[m / LR];
    int gr[16], gc[16];
    const int nr = axis_groups(first_tap[2 * m + 1], gr), nc = axis_groups(first_tap[2 * m], gc);
    for (int a = 0; a < nr; ++a)
      for (int b = 0; b < nc; ++b) gcnt[(frame * gps + gr[a]) * gps + gc[b]]++;
  }
  std::vector<int> glen(ngroup);
  for (size_t g = 0; g < ngroup; ++g) glen[g] = (gcnt[g] + kSpreadListPad - 1) / kSpreadListPad * kSpreadListPad;
  std::vector<int> gorder;
  gorder.reserve(ngroup);
  static_assert(kGridBlock % kSpreadGroup == 0, "a group lies in one grid block");
  auto in_use = [&](int t, int gr, int gc) {
    return p.grid_used_h.empty() || (p.grid_used_h[(size_t)t * gps + gc] >> (gr * G / kGridBlock) & 1);
  };
  for (int t = 0; t < p.T; ++t)
    for (int pr = 0; pr < gps / PG; ++pr)
      for (int pc = 0; pc < gps / PG; ++pc)
        for (int r = 0; r < PG; ++r)
          for (int c = 0; c < PG; ++c)
            if (in_use(t, pr * PG + r, pc * PG + c)) gorder.push_back((t * gps + pr * PG + r) * gps + pc * PG + c);
  const size_t nlisted = gorder.size();
  std::vector<int> item_of(ngroup), first(ngroup);
  struct ItemSec { size_t offs, wts; };
  std::vector<ItemSec> secs;
  auto words = [](long ng, long ne) { return ((ng + 1) & ~1L) + ne / 2 + 2 * ne; };
  size_t i = 0;
  while (i < nlisted) {
    size_t j = i;
    long cost = 0, nent = 0;
    while (j < nlisted) {
      const int c = glen[gorder[j]];
      if (words((long)(j + 1 - i), nent + c) > kSpreadStageInt2) {
        if (j == i) return false;  // one group exceeds a stage
        break;
      }
      nent += c;
      cost += c + kSpreadGroupCost;
      ++j;
      if (cost >= kSpreadGroupItemCost) break;
    }
    const long ng = (long)(j - i), ngp = (ng + 1) & ~1L;
    const size_t at = blob.size();
    if (at + (size_t)words(ng, nent) > 0x7fffffffULL) return false;
    sitems.push_back(make_int4((int)at, (int)ng, (int)nent, (int)words(ng, nent)));
    secs.push_back({at + (size_t)ngp, at + (size_t)ngp + (size_t)nent / 2});
    blob.resize(at + (size_t)words(ng, nent), make_int2(0, 0));
    {
      int* offs = reinterpret_cast<int*>(&blob[secs.back().offs]);
      for (long q = 0; q < nent; ++q) offs[q] = (int)((size_t)p.M * p.cs);  // padding: the zero row
    }
    long e = 0;
    for (size_t q = i; q < j; ++q) {
      const int g = gorder[q];
      item_of[g] = (int)sitems.size() - 1;
      first[g] = (int)e;
      e += glen[g];
      const int t = g / (gps * gps), gr = (g / gps) % gps, gc = g % gps;
      blob[at + (q - i)] = make_int2((int)(((size_t)t * n + (size_t)gr * G) * n + (size_t)gc * G), (int)e);
    }
    i = j;
  }
  std::vector<int> cursor(ngroup, 0);
  for (size_t m = 0; m < (size_t)p.M; ++m) {
    const size_t frame = (size_t)p.blade_frame[m / LR];
    const int r0 = first_tap[2 * m + 1], c0 = first_tap[2 * m];
    int gr[16], gc[16];
    const int nr = axis_groups(r0, gr), nc = axis_groups(c0, gc);
    for (int a = 0; a < nr; ++a)
      for (int b = 0; b < nc; ++b) {
        const int g = (int)((frame * gps + gr[a]) * gps + gc[b]);
        const ItemSec& sec = secs[item_of[g]];
        const size_t e = (size_t)first[g] + cursor[g]++;
        float w[4];
        for (int ii = 0; ii < G; ++ii)
          for (int jj = 0; jj < G; ++jj) {
            const int da = (gr[a] * G + ii - r0 + n) % n, db = (gc[b] * G + jj - c0 + n) % n;
            w[ii * G + jj] = (da < W && db < W) ? (float)(wd[m * 2 * W + W + da] * wd[m * 2 * W + db]) : 0.f;
          }
        reinterpret_cast<int*>(&blob[sec.offs])[e] = (int)(m * (size_t)p.cs);
        std::memcpy(&blob[sec.wts + 2 * e], w, sizeof(w));
      }
  }
  return true;
}

// Grid blocks (kGridBlock rows of two adjacent columns) that some sample's
// W x W footprint meets.
void mark_used_blocks(Plan& p, const std::vector<int>& first_tap) {
  const int n = p.n, W = p.W;
  static_assert(kGridBlock >= 8, "a footprint's rows meet at most two blocks");
  p.grid_used_h.assign((size_t)p.T * (n / 2), 0);
  const size_t LR = (size_t)p.L * p.R;
  for (size_t m = 0; m < (size_t)p.M; ++m) {
    uint64_t* used = &p.grid_used_h[(size_t)p.blade_frame[m / LR] * (n / 2)];
    const int r0 = first_tap[2 * m + 1], c0 = first_tap[2 * m];
    const uint64_t rows = 1ull << (r0 / kGridBlock) | 1ull << ((r0 + W - 1) % n / kGridBlock);
    for (int b = 0; b < W; ++b) used[(c0 + b) % n / 2] |= rows;
  }
  size_t count = 0;
  for (uint64_t u : p.grid_used_h) count += (size_t)__builtin_popcountll(u);
  p.grid_sparse = 2 * count < p.grid_used_h.size() * (size_t)(n / kGridBlock);
}

// Interpolation tiles and their work items: samples sorted by (frame, TR x
// TC-cell tile of their first tap), ascending m within a tile; every non-empty
// tile's run is cut into items of at most kInterpItem samples.  One CTA per
// item stages the tile plus its (W - 1)-cell halo in shared memory.  Static
// balance over `ctas` persistent CTAs: longest item first to the least loaded
// CTA, with an item's cost its shared-memory traffic (W^2 taps of cs bins per
// sample plus the staged tile); each CTA's items are then stored contiguously,
// in tile order.
void build_tiles(const Plan& p, const std::vector<int>& first_tap, int ctas, std::vector<int>& order,
                 std::vector<int4>& items, std::vector<int>& cta_off) {
  const int TR = interp_tile_rows(p.cs, p.W), TC = interp_tile_cols(p.cs);
  const int nrt = (p.n + TR - 1) / TR, nct = p.n / TC;  // tiles per column / per row of the grid
  const size_t ntile = (size_t)p.T * nrt * nct, LR = (size_t)p.L * p.R;
  auto tile_of = [&](size_t m) {
    const size_t frame = (size_t)p.blade_frame[m / LR];
    return (frame * nrt + first_tap[2 * m + 1] / TR) * nct + first_tap[2 * m] / TC;
  };
  std::vector<int> cnt(ntile + 1, 0);
  for (size_t m = 0; m < (size_t)p.M; ++m) cnt[tile_of(m) + 1]++;
  for (size_t t = 0; t < ntile; ++t) cnt[t + 1] += cnt[t];
  std::vector<int4> by_tile;
  for (size_t t = 0; t < ntile; ++t) {
    // a tile's run in ceil(c / kInterpItem) items of nearly equal size
    const int c = cnt[t + 1] - cnt[t];
    const int parts = (c + kInterpItem - 1) / kInterpItem;
    for (int q = 0, s = cnt[t]; q < parts; ++q) {
      const int sz = c / parts + (q < c % parts ? 1 : 0);
      by_tile.push_back(make_int4((int)t, s, sz, 0));
      s += sz;
    }
  }
  order.resize(p.M);
  for (size_t m = 0; m < (size_t)p.M; ++m) order[cnt[tile_of(m)]++] = (int)m;
  const int P = std::max(1, std::min(ctas, (int)by_tile.size()));
  const long tile_cost = (long)(TR + p.W - 1) * (TC + p.W - 1) * p.cs / 16;
  auto cost = [&](const int4& it) { return (long)it.z * p.W * p.W * p.cs / 16 + tile_cost; };
  std::vector<int> idx(by_tile.size());
  for (size_t i = 0; i < idx.size(); ++i) idx[i] = (int)i;
  std::stable_sort(idx.begin(), idx.end(), [&](int a, int b) { return cost(by_tile[a]) > cost(by_tile[b]); });
  std::vector<long> load(P, 0);
  std::vector<std::vector<int>> own(P);
  for (int i : idx) {
    const int best = (int)(std::min_element(load.begin(), load.end()) - load.begin());
    load[best] += cost(by_tile[i]);
    own[best].push_back(i);
  }
  items.clear();
  cta_off.assign(P + 1, 0);
  for (int c = 0; c < P; ++c) {
    std::sort(own[c].begin(), own[c].end());
    for (int i : own[c]) items.push_back(by_tile[i]);
    cta_off[c + 1] = (int)items.size();
  }
}

// Modelled cost of an interpolation item in clock cycles of an SM, from fits
// to the CTAs' own clocks at the static (32 bins), dynamic (16) and 64-bin
// configurations: an item's turn round the warps, its quads, and the copies of
// the rows it adds to the ring (from L2 or, where the used part of the grid
// outgrows it, from DRAM).
long quad_cost(int quads, int new_rows, int cs, bool grid_in_l2) {
  return (cs == 64 ? 5000 : 1600) + 140 * (long)quads + (long)new_rows * (grid_in_l2 ? 60 : 250);
}

// Interpolation quads (prop_internal.cuh) and their work items.  A quad's
// anchor is the cell of its window's first row and column; quads are ordered
// by frame, strip of quad_cols(cs) columns, first row and sample index, and
// a strip's run is cut into items of at most quad_item(cs) quads that start
// within quad_span(cs, W) rows.  A CTA takes a contiguous run of items, so that
// it walks down a strip and an item adds only its last rows to those of the
// item before; the runs are cut at equal shares of the modelled cost.
void build_quads(const Plan& p, const std::vector<int>& first_tap, const std::vector<double>& wd, int ctas,
                 std::vector<float4>& quads, std::vector<int4>& items, std::vector<int>& cta_off) {
  const int n = p.n, W = p.W, UW = quad_window(W), REC = quad_record(W), TC = quad_cols(p.cs);
  const int nstrip = (n + TC - 1) / TC;
  struct Quad {
    int m[4], d1[4], d2[4], c0, r0, j0, key;
  };
  std::vector<Quad> qs;
  for (int b = 0; b < p.B; ++b)
    for (int l = 0; l < p.L; l += 2)
      for (int j = 0; j < p.R; j += 2) {
        Quad q{};
        int ref = -1, lo1 = 0, lo2 = 0;
        for (int s = 0; s < 4; ++s) {
          const int ls = l + s / 2, js = j + s % 2;
          q.m[s] = ls < p.L && js < p.R ? (b * p.L + ls) * p.R + js : -1;
          if (q.m[s] < 0) continue;
          if (ref < 0) ref = q.m[s];
          // tap distances from the first sample's, on the circle
          auto dist = [&](int axis) {
            const int d = first_tap[2 * (size_t)q.m[s] + axis] - first_tap[2 * (size_t)ref + axis];
            return ((d + n / 2) % n + n) % n - n / 2;
          };
          q.d1[s] = dist(0);
          q.d2[s] = dist(1);
          lo1 = std::min(lo1, q.d1[s]);
          lo2 = std::min(lo2, q.d2[s]);
        }
        for (int s = 0; s < 4; ++s) q.d1[s] -= lo1, q.d2[s] -= lo2;
        q.c0 = (first_tap[2 * (size_t)ref] + lo1 + n) % n;
        q.r0 = (first_tap[2 * (size_t)ref + 1] + lo2 + n) % n;
        q.j0 = j;
        q.key = p.blade_frame[b] * nstrip + q.c0 / TC;
        qs.push_back(q);
      }
  std::vector<int> idx(qs.size());
  for (size_t i = 0; i < idx.size(); ++i) idx[i] = (int)i;
  std::stable_sort(idx.begin(), idx.end(), [&](int x, int y) {
    return qs[x].key != qs[y].key ? qs[x].key < qs[y].key : qs[x].r0 < qs[y].r0;
  });
  std::vector<int> row0(qs.size());  // first row of each quad's item
  std::vector<long> upto;            // cost up to and with each item
  long total = 0;
  // Small problems take smaller items (of whole units), so that every CTA has
  // one: 5 blades of 8 x 32 samples in 8 bins 12.3 -> 8.6 us, 8 blades of 16 x
  // 64 samples 15.8 -> 13.8 us.
  const int per = quad_per_warp(p.cs), fair = ((int)qs.size() + ctas - 1) / ctas;
  const int span = quad_span(p.cs, W), most = std::min(quad_item(p.cs), (fair + per - 1) / per * per);
  size_t blocks = 0;
  for (uint64_t u : p.grid_used_h) blocks += (size_t)__builtin_popcountll(u);
  const bool in_l2 = blocks * 2 * kGridBlock * p.cs * sizeof(float2) < (size_t)100 << 20;
  for (size_t i = 0; i < idx.size();) {
    const Quad& q0 = qs[idx[i]];
    size_t e = i;
    while (e < idx.size() && (int)(e - i) < most && qs[idx[e]].key == q0.key && qs[idx[e]].r0 < q0.r0 + span)
      row0[e++] = q0.r0;
    const int rows = qs[idx[e - 1]].r0 - q0.r0 + UW;
    const int have = items.empty() || items.back().x != q0.key
                         ? 0
                         : std::max(0, (items.back().w & 0xffff) + (items.back().w >> 16) - q0.r0);
    total += quad_cost((int)(e - i), rows - std::min(rows, have), p.cs, in_l2);
    upto.push_back(total);
    items.push_back(make_int4(q0.key, (int)i, (int)(e - i), q0.r0 | rows << 16));
    i = e;
  }
  quads.assign(qs.size() * REC, make_float4(0.f, 0.f, 0.f, 0.f));
  for (size_t i = 0; i < idx.size(); ++i) {
    const Quad& q = qs[idx[i]];
    float* w = reinterpret_cast<float*>(&quads[i * REC]);
    int* tail = reinterpret_cast<int*>(&quads[i * REC + 2 * UW]);
    int rows = 0, cols = 0;
    for (int s = 0; s < 4; ++s) {
      tail[s] = q.m[s];
      if (q.m[s] < 0) continue;
      for (int a = 0; a < W; ++a) {
        w[4 * (q.d1[s] + a) + s] = (float)wd[(size_t)q.m[s] * 2 * W + a];
        w[4 * (UW + q.d2[s] + a) + s] = (float)wd[(size_t)q.m[s] * 2 * W + W + a];
      }
      rows = std::max(rows, q.d2[s] + W);
      cols = std::max(cols, q.d1[s] + W);
    }
    tail[4] = q.r0 - row0[i];
    tail[5] = q.c0 % TC;
    tail[6] = q.j0;
    tail[7] = rows | cols << 8;
  }
  const int P = std::max(1, std::min(ctas, (int)items.size()));
  cta_off.assign(P + 1, (int)items.size());
  cta_off[0] = 0;
  for (int c = 1, at = 0; c < P; ++c) {
    // the cut nearest to c shares of the cost, with an item left for every CTA
    const long want = total * c / P;
    ++at;
    while (at < (int)items.size() - (P - c) && upto[at - 1] + (upto[at] - upto[at - 1]) / 2 < want) ++at;
    cta_off[c] = at;
  }
}

// What the two interpolations of the bin strides 8 to 64 cost, in ns of a CTA:
// tiles an item, a round of the warps over an item's samples (width 8; the
// latency of one), a round's worth of samples (width 8; its shared-memory
// wavefronts); quads an item, a unit (what a warp takes at once; width 8), a
// grid row added to the ring (its width in cells as at width 8), and the
// difference of the launches (the quads' 227 KB of shared memory do not overlap
// the kernel before).  Fitted to the times of both, forward passes replayed from
// a graph and iterations of a reconstruction, at 1150 geometries (N = 16 to 512,
// 1 to 32 frames, 1 to 64 lines, both widths): the plan's longest CTA decides,
// as every CTA runs alone on its SM.
struct InterpModel {
  int t_item, t_round, t_samples, q_item, q_unit, q_row, q_launch;
};
constexpr InterpModel interp_model(int cs) {
  return cs == 8    ? InterpModel{1630, 860, 2700, 780, 234, 160, -850}
         : cs == 16 ? InterpModel{1420, 750, 1520, 1170, 158, 121, 0}
         : cs == 32 ? InterpModel{1090, 570, 1710, 540, 170, 122, 450}
                    : InterpModel{730, 1130, 1070, 1790, 251, 72, 1700};
}
// Modelled times of a cut: of its longest CTA and of all of them together.
struct InterpTime {
  double longest = 0, total = 0;
  void add(double t) {
    longest = std::max(longest, t);
    total += t;
  }
};
InterpTime tiles_time(const Plan& p, const std::vector<int4>& items, const std::vector<int>& cta_off) {
  const InterpModel k = interp_model(p.cs);
  const int round = kTileWarps * tile_samples_per_warp(p.cs);
  InterpTime time;
  for (size_t c = 0; c + 1 < cta_off.size(); ++c) {
    long samples = 0, rounds = 0;
    for (int i = cta_off[c]; i < cta_off[c + 1]; ++i) {
      samples += items[i].z;
      rounds += (items[i].z + round - 1) / round;
    }
    time.add((double)k.t_item * (cta_off[c + 1] - cta_off[c]) + k.t_round * p.W / 8.0 * rounds +
             k.t_samples * (p.W * p.W / 64.0) * samples / round);
  }
  return time;
}
InterpTime quads_time(const Plan& p, const std::vector<int4>& items, const std::vector<int>& cta_off) {
  const InterpModel k = interp_model(p.cs);
  const double unit = k.q_unit * (quad_window(p.W) * quad_window(p.W) / 121.0);
  const double row = (double)k.q_row * quad_row_bytes(p.cs, p.W) / quad_row_bytes(p.cs, 8);
  InterpTime time;
  for (size_t c = 0; c + 1 < cta_off.size(); ++c) {
    long units = 0, rows = 0;
    for (int i = cta_off[c]; i < cta_off[c + 1]; ++i) {
      const int4 it = items[i];
      const int r0 = it.w & 0xffff, nr = it.w >> 16;
      units += (it.z + quad_per_warp(p.cs) - 1) / quad_per_warp(p.cs);
      const bool on = i > cta_off[c] && items[i - 1].x == it.x;  // the strip goes on: only new rows
      rows += nr - std::min(nr, on ? std::max(0, (items[i - 1].w & 0xffff) + (items[i - 1].w >> 16) - r0) : 0);
    }
    time.add((double)k.q_item * (cta_off[c + 1] - cta_off[c]) + unit * units + row * rows);
  }
  time.longest += k.q_launch;
  return time;
}

struct DevAlloc {
  Plan* p;
  size_t* counter;
  template <class T>
  prop_status operator()(T** ptr, size_t count, const char* what) {
    *ptr = nullptr;
    if (count == 0) count = 1;
    cudaError_t e = plan_dev_alloc(p, (void**)ptr, count * sizeof(T));
    if (e != cudaSuccess) {
      cudaGetLastError();
      *ptr = nullptr;
      return fail(PROP_ERR_OOM, std::string("cudaMalloc failed for ") + what + ": " +
                                    cudaGetErrorString(e));
    }
    *counter += count * sizeof(T);
    return PROP_OK;
  }
};

template <class T>
prop_status upload(T* dst, const std::vector<T>& src) {
  PROP_CUDA(cudaMemcpy(dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice));
  return PROP_OK;
}

}  // namespace

cudaError_t plan_dev_alloc(Plan* p, void** ptr, size_t bytes) {
  return p->alloc ? p->alloc->allocate(ptr, bytes) : cudaMalloc(ptr, bytes);
}

void plan_dev_free(Plan* p, void* ptr) {
  if (!ptr) return;
  if (p->alloc)
    p->alloc->release(ptr);
  else
    cudaFree(ptr);
}

void plan_free(Plan* p) {
  if (!p) return;
  void* ptrs[] = {p->kb_idx, p->kb_w, p->phase, p->deapod, p->twiddle, p->blade_frame_d,
                  p->order, p->quads, p->tile_cut.items, p->tile_cut.off, p->quad_cut.items, p->quad_cut.off, p->grid_used, p->sitems, p->sitem_cta_off, p->spread_claim, p->sblob, p->contrib, p->grid, p->rows,
                  p->resid, p->grad, p->status_dev,
                  p->vol2, p->adam_m, p->adam_v, p->loss_dev, p->scalars,
                  p->red_interp.partials, p->red_interp.counter, p->red_tv.partials,
                  p->red_tv.counter, p->stage_y, p->stage_v, p->proj_shift, p->proj_mask, p->proj_twiddle,
                  p->proj_img, p->proj_k, p->proj_kg, p->proj_g, p->proj_yimg, p->proj_const,
                  p->red_proj_k.partials, p->red_proj_k.counter, p->red_proj_u.partials, p->red_proj_u.counter,
                  p->psnr_scratch, p->kp_work};
  for (void* q : ptrs) plan_dev_free(p, q);
  if (p->host_words) cudaFreeHost(p->host_words);
  for (cudaEvent_t e : p->ev_pool) cudaEventDestroy(e);
  for (auto& v : p->ev_rec)
    for (auto& pr : v) {
      cudaEventDestroy(pr.first);
      cudaEventDestroy(pr.second);
    }
  delete p;
}

prop_status plan_build(const prop_plan_desc* d, Plan** out, DeviceAllocator* alloc) {
  if (!d || !out) return fail(PROP_ERR_INVALID_ARG, "plan_create: null argument");
  *out = nullptr;
  const int N = d->n;
  if (N < 16 || N > 512 || N % 8 != 0 || !fft_size_supported(2 * N))
    return fail(PROP_ERR_INVALID_ARG,
                "plan_create: n must be a multiple of 8 in [16, 512] with 2n = 2^a 3^b (n = " +
                    std::to_string(N) + ")");
  if (d->nf < 1 || d->nf > 4096) return fail(PROP_ERR_INVALID_ARG, "plan_create: nf out of range");
  if (d->nblades < 1 || d->lines < 1 || d->readout < 1)
    return fail(PROP_ERR_INVALID_ARG, "plan_create: nblades, lines and readout must be >= 1");
  if ((long long)d->nblades * d->lines * d->readout > (1LL << 30))
    return fail(PROP_ERR_INVALID_ARG, "plan_create: too many samples");
  if ((long long)d->nblades * d->lines * d->readout * kMaxChunk >= (1LL << 31))
    return fail(PROP_ERR_INVALID_ARG, "plan_create: too many samples for 32-bit spread offsets");
  if (d->nframes < 1) return fail(PROP_ERR_INVALID_ARG, "plan_create: nframes must be >= 1");
  if (!d->delta || !d->theta) return fail(PROP_ERR_INVALID_ARG, "plan_create: delta/theta is NULL");
  if (d->kb_width != 0 && d->kb_width != 6 && d->kb_width != 8)
    return fail(PROP_ERR_INVALID_ARG, "plan_create: kb_width must be 0 (= 6), 6 or 8");
  if (d->bin_chunk < 0 || d->bin_chunk > kMaxChunk)
    return fail(PROP_ERR_INVALID_ARG, "plan_create: bin_chunk must be in [0, 64]");
  if (d->row_kernel < 0 || d->row_kernel > 2)
    return fail(PROP_ERR_INVALID_ARG, "plan_create: row_kernel must be 0, 1 or 2");
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || d->device < 0 || d->device >= ndev) {
    cudaGetLastError();
    return fail(PROP_ERR_INVALID_ARG, "plan_create: no such CUDA device");
  }
  for (int f = 0; f < d->nf; ++f)
    if (!std::isfinite(d->delta[f])) return fail(PROP_ERR_INVALID_ARG, "plan_create: delta not finite");
  for (int b = 0; b < d->nblades; ++b) {
    if (!std::isfinite(d->theta[b])) return fail(PROP_ERR_INVALID_ARG, "plan_create: theta not finite");
    if (d->blade_frame && (d->blade_frame[b] < 0 || d->blade_frame[b] >= d->nframes))
      return fail(PROP_ERR_INVALID_ARG, "plan_create: blade_frame out of range");
  }

  Plan* p = new (std::nothrow) Plan();
  if (!p) return fail(PROP_ERR_OOM, "plan_create: host allocation failed");
  p->alloc = alloc;
  p->N = N;
  p->n = 2 * N;
  p->Nf = d->nf;
  p->B = d->nblades;
  p->L = d->lines;
  p->R = d->readout;
  p->T = d->nframes;
  p->M = p->B * p->L * p->R;
  p->device = d->device;
  p->W = d->kb_width == 0 ? kKbWidthDefault : d->kb_width;
  p->chunk = d->bin_chunk == 0 ? std::min(p->Nf, kMaxChunk) : std::min(d->bin_chunk, p->Nf);
  p->nchunks = (p->Nf + p->chunk - 1) / p->chunk;
  p->cs = p->chunk + (p->chunk & 1);  // even stride: staged grid rows are 16-byte runs
  p->theta.assign(d->theta, d->theta + p->B);
  p->delta.assign(d->delta, d->delta + p->Nf);
  p->blade_frame.assign(p->B, 0);
  if (d->blade_frame) p->blade_frame.assign(d->blade_frame, d->blade_frame + p->B);

  DeviceGuard guard(p->device);
  if (!guard.ok) {
    plan_free(p);
    return fail(PROP_ERR_CUDA, "plan_create: cudaSetDevice failed");
  }
  if (cudaDeviceGetAttribute(&p->num_sms, cudaDevAttrMultiProcessorCount, p->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&p->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, p->device) != cudaSuccess) {
    cudaGetLastError();
    plan_free(p);
    return fail(PROP_ERR_CUDA, "plan_create: device attribute query failed");
  }

  const int n = p->n;
  const int Wi = p->W;
  const double W = Wi, sigma = 2.0;
  const double beta = M_PI * std::sqrt((W / sigma) * (W / sigma) * (sigma - 0.5) * (sigma - 0.5) - 0.8);
  const double i0b = bessel_i0(beta);

  auto psi = [&](double t) {
    double a = 2.0 * t / W;
    double r = 1.0 - a * a;
    if (r < 0.0) return 0.0;
    return bessel_i0(beta * std::sqrt(r)) / i0b;
  };

  // Per-sample grid indices and weights.
  std::vector<uint32_t> kb_idx(p->M);
  const int wq = Wi / 2;  // float4 per sample
  std::vector<float4> kb_w((size_t)p->M * wq);
  std::vector<int> first_tap(2 * (size_t)p->M);
  std::vector<double> wd((size_t)p->M * 2 * Wi);  // FP64 weights: w1[W] then w2[W]
  for (int b = 0; b < p->B; ++b) {
    const double c = std::cos(p->theta[b]), s = std::sin(p->theta[b]);
    for (int l = 0; l < p->L; ++l) {
      const double kp = ((double)l - p->L / 2.0) / N;
      for (int j = 0; j < p->R; ++j) {
        const double kr = ((double)j - p->R / 2.0) / N;
        const double k[2] = {kr * c - kp * s, kr * s + kp * c};
        const size_t m = ((size_t)b * p->L + l) * p->R + j;
        float w[16];
        int base[2];
        for (int a = 0; a < 2; ++a) {
          double u = n * k[a];
          u -= n * std::floor(u / n);
          if (u >= n) u -= n;
          if (u < 0) u = 0;
          const double fl = std::floor(u);
          const double fr = u - fl;
          const int h = Wi / 2 - 1;  // taps floor(u) - h .. floor(u) + W/2
          base[a] = ((int)fl - h + n) % n;
          for (int q = 0; q < Wi; ++q) {
            const double v = psi(fr + h - q);
            wd[m * 2 * Wi + a * Wi + q] = v;
            w[a * Wi + q] = (float)v;
          }
        }
        kb_idx[m] = (uint32_t)base[0] | ((uint32_t)base[1] << 16);
        first_tap[2 * m] = base[0];
        first_tap[2 * m + 1] = base[1];
        for (int q = 0; q < wq; ++q)
          kb_w[(size_t)wq * m + q] = make_float4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
      }
    }
  }

  // Deapodisation along one axis.
  std::vector<float> deapod(N);
  for (int i = 0; i < N; ++i) {
    const double xi = (double)(i - N / 2) / n;
    const double a = M_PI * W * xi;
    const double z2 = beta * beta - a * a;
    double ft;
    if (z2 > 0) {
      const double z = std::sqrt(z2);
      ft = W * std::sinh(z) / z;
    } else if (z2 < 0) {
      const double z = std::sqrt(-z2);
      ft = W * std::sin(z) / z;
    } else {
      ft = W;
    }
    deapod[i] = (float)(i0b / ft);
  }

  // Displacement phase per readout sample and bin.
  std::vector<float2> phase((size_t)p->R * p->Nf);
  for (int j = 0; j < p->R; ++j) {
    const double kr = ((double)j - p->R / 2.0) / N;
    for (int f = 0; f < p->Nf; ++f) {
      double arg = kr * p->delta[f];
      arg -= std::nearbyint(arg);
      phase[(size_t)j * p->Nf + f] = make_float2((float)std::cos(2 * M_PI * arg),
                                                 (float)-std::sin(2 * M_PI * arg));
    }
  }

  std::vector<float2> tw(n);
  for (int q = 0; q < n; ++q)
    tw[q] = make_float2((float)std::cos(2 * M_PI * q / n), (float)-std::sin(2 * M_PI * q / n));

  // Interpolation work items.  At the bin strides 8 to 64 the plan takes quads
  // or tiles, whichever the model has faster (the results are the same bit for
  // bit).  Quads win where samples are dense (the static benchmark's operator,
  // 32 bins: a forward pass 92 -> 85 us) or crowd into few tiles (one frame of 48
  // blades of 4 lines at N = 32, 64 bins: 43.7 -> 14 us); tiles where a frame has
  // few samples (32 frames of 2 x 4 lines at N = 16, 64 bins: 32.0 -> 26.3 us),
  // where one line a blade leaves half of a quad empty (192^2 x 64 bins, 32
  // frames: 104 -> 64 us of interpolation) and with 64 bins at width 8 unless the
  // samples crowd (one scan of 16 blades, N = 256: 168 -> 123 us).  Over the
  // fitted geometries the rule's forward pass is 0.2 % slower than that of the
  // better of the two; quads alone were 3.4 %, tiles 23 %.
  // A batch shares the CTAs out over its plans, so that a plan's share counts, not
  // its longest CTA: it takes quads where they cost less in total, and a plan keeps
  // both where the two differ.  At 8 and 16 bins, where a batch of both kinds was 5
  // to 8 % slower than one of quads (four plans of 96^2 x 16 bins: 884 and 814 us),
  // tiles have to cost half as much in total (24^2 x 16 bins: 245 and 267 us).
  const size_t LR = (size_t)p->L * p->R;
  std::vector<int> order, tile_off, quad_off;
  std::vector<int4> tile_items, quad_items;
  std::vector<float4> quads;
  build_tiles(*p, first_tap, p->num_sms, order, tile_items, tile_off);
  if (quad_stride(p->cs)) {
    mark_used_blocks(*p, first_tap);
    build_quads(*p, first_tap, wd, p->num_sms, quads, quad_items, quad_off);
    const InterpTime tt = tiles_time(*p, tile_items, tile_off), qt = quads_time(*p, quad_items, quad_off);
    p->lone_quads = qt.longest < tt.longest;
    if (!p->lone_quads && tt.total < (p->cs <= 16 ? 0.5 : 1.0) * qt.total) {
      quads.clear();
      quad_items.clear();
      quad_off.clear();
    }
    if (p->lone_quads) {
      kb_idx.clear();
      kb_w.clear();
      order.clear();
      tile_items.clear();
      tile_off.clear();
    }
  }
  if (!p->lone_quads) {
    // The tile kernels read the per-sample tables in item order, so that an
    // item's metadata is one contiguous run.
    std::vector<uint32_t> idx_s(p->M);
    std::vector<float4> w_s(kb_w.size());
    for (size_t i = 0; i < (size_t)p->M; ++i) {
      const size_t m = (size_t)order[i];
      idx_s[i] = kb_idx[m];
      for (int q = 0; q < wq; ++q) w_s[i * wq + q] = kb_w[m * wq + q];
    }
    kb_idx.swap(idx_s);
    kb_w.swap(w_s);
  }

  // Spread gather lists: for every (frame, cell) the samples whose W x W
  // footprint covers the cell, as (phased-residual offset m * cs, weight
  // w2[a] w1[b]) in ascending m.  The weight is formed in FP64 from the same
  // factors the interpolation applies, so the spread is its exact transpose.
  // Cells are listed in patch-major order (frame, 8x8-cell patch, row-major in
  // the patch) and cut into work items of about equal work (list entries plus
  // a fixed cost per written cell); patch order keeps the residual rows an
  // item reads within a small region of k-space.
  std::vector<int4> sitems;
  std::vector<int2> blob;
  const int2 pad_entry = make_int2((int)((size_t)p->M * p->cs), 0);
  p->spread_grouped = quad_stride(p->cs) && build_group_lists(*p, first_tap, wd, sitems, blob);
  if (!p->spread_grouped) {
  p->grid_used_h.clear();  // the cell lists fill the whole grid
  p->grid_sparse = false;
  sitems.clear();
  blob.clear();
  const size_t ncell = (size_t)p->T * n * n;
  std::vector<int> cell_cnt(ncell, 0);
  auto cell_of = [&](size_t m, int a, int b) {
    const size_t frame = (size_t)p->blade_frame[m / LR];
    const int r = (first_tap[2 * m + 1] + a) % n, c = (first_tap[2 * m] + b) % n;
    return (frame * n + r) * n + c;
  };
  for (size_t m = 0; m < (size_t)p->M; ++m)
    for (int a = 0; a < Wi; ++a)
      for (int b = 0; b < Wi; ++b) cell_cnt[cell_of(m, a, b)]++;
  std::vector<int> cell_ids(ncell);
  {
    const int pps = n / kSpreadPatch;
    size_t i = 0;
    for (int t = 0; t < p->T; ++t)
      for (int pr = 0; pr < pps; ++pr)
        for (int pc = 0; pc < pps; ++pc)
          for (int r = 0; r < kSpreadPatch; ++r)
            for (int c = 0; c < kSpreadPatch; ++c)
              cell_ids[i++] = (int)(((size_t)t * n + pr * kSpreadPatch + r) * n + pc * kSpreadPatch + c);
  }
  // Work items: runs of consecutive cells (patch-major order) of about equal
  // work (list entries plus a fixed cost per written cell), each stored as
  // one contiguous blob that a CTA stages into shared memory with a single
  // bulk copy:
  //   int2 cells[ncells, rounded up to even]: (cell index, end of its list
  //        relative to the item's first entry)
  //   int2 entries[nent]: the lists, one after the other
  // Every list is padded to a multiple of kSpreadListPad entries with
  // (row M, weight 0): row M of the phased-residual buffer is kept zero, so
  // a padding entry adds an exact zero and the gather runs unpredicated.  A
  // cell whose list alone exceeds the staging capacity forms an item of its
  // own and the plan then gathers from global memory.
  std::vector<int> cell_first(ncell + 1, 0);  // cell -> first entry in the item's entries
  {
    auto padded = [](int c) { return (c + kSpreadListPad - 1) / kSpreadListPad * kSpreadListPad; };
    size_t i = 0;
    while (i < ncell) {
      // choose [i, j)
      size_t j = i;
      long cost = 0, nent = 0;
      while (j < ncell) {
        const int c = padded(cell_cnt[cell_ids[j]]);
        const long ncp = (long)((j + 1 - i + 1) & ~(size_t)1);
        if (j > i && ncp + nent + c > kSpreadStageInt2) break;  // would overflow the stage
        nent += c;
        cost += c + kSpreadCellCost;
        ++j;
        if (cost >= kSpreadItemCost) break;
      }
      const size_t ncells = j - i, ncp = (ncells + 1) & ~(size_t)1;
      if ((long)ncp + nent > kSpreadStageInt2) p->spread_staged = false;  // longer than a stage: read from global
      if (blob.size() + ncp + nent > 0x7fffffffULL) {
        plan_free(p);
        return fail(PROP_ERR_INVALID_ARG, "plan_create: spread lists exceed 2^31 entries");
      }
      sitems.push_back(make_int4((int)blob.size(), (int)ncells, (int)nent, (int)(ncp + nent)));
      const size_t cells_at = blob.size(), ent_at = cells_at + ncp;
      blob.resize(ent_at + nent, pad_entry);
      long e = 0;
      for (size_t q = i; q < j; ++q) {
        const int cid = cell_ids[q];
        cell_first[cid] = (int)(ent_at + e);
        e += padded(cell_cnt[cid]);
        blob[cells_at + (q - i)] = make_int2(cid, (int)e);
      }
      if (ncp > ncells) blob[cells_at + ncells] = make_int2(0, (int)e);
      i = j;
    }
  }
  for (size_t m = 0; m < (size_t)p->M; ++m)
    for (int a = 0; a < Wi; ++a)
      for (int b = 0; b < Wi; ++b) {
        const float w = (float)(wd[m * 2 * Wi + Wi + a] * wd[m * 2 * Wi + b]);
        int wbits;
        std::memcpy(&wbits, &w, sizeof(float));
        blob[cell_first[cell_of(m, a, b)]++] = make_int2((int)(m * (size_t)p->cs), wbits);
      }
  }
  // every item's blob (its word count is the staged copy's size) lies in the
  // list array, and a staged item fits a stage
  for (const int4& it : sitems) {
    const bool staged = p->spread_grouped || p->spread_staged;
    if (it.x < 0 || it.w < 0 || (size_t)it.x + (size_t)it.w > blob.size() || (staged && it.w > kSpreadStageInt2)) {
      plan_free(p);
      return fail(PROP_ERR_INVALID_ARG, "plan_create: inconsistent spread lists");
    }
  }
  p->n_sitems = (int)sitems.size();
  p->spread_entries = blob.size();
  // Schedule of the spread items over the staged kernel's persistent CTAs
  // (two per SM).  With few items per CTA, a plan-time balance (longest
  // first to the least loaded CTA, each CTA's items then in k-space order so
  // that consecutive items share residual rows in L1) and CTA c takes
  // [off[c], off[c + 1]).  With many (kSpreadClaimMinItems per CTA or more),
  // grouped lists keep the items in k-space order and the CTAs claim them
  // from a device counter, so each CTA's share follows the items' measured
  // cost.
  std::vector<int> scta_off;
  {
    const int P = std::max(1, std::min(kSpreadCtasPerSm * p->num_sms, p->n_sitems));
    p->spread_claimed = p->spread_grouped && p->n_sitems >= kSpreadClaimMinItems * P;
    if (p->spread_claimed) {
      scta_off = {0, p->n_sitems};
    } else {
      auto cost = [&](const int4& it) {
        return (long)it.z + (long)it.y * (p->spread_grouped ? kSpreadGroupCost : kSpreadCellCost);
      };
      std::vector<int> idx(sitems.size());
      for (size_t q = 0; q < idx.size(); ++q) idx[q] = (int)q;
      std::stable_sort(idx.begin(), idx.end(), [&](int a, int b) { return cost(sitems[a]) > cost(sitems[b]); });
      std::vector<long> load(P, 0);
      std::vector<std::vector<int>> own(P);
      for (int q : idx) {
        int best = 0;
        for (int c = 1; c < P; ++c)
          if (load[c] < load[best]) best = c;
        load[best] += cost(sitems[q]);
        own[best].push_back(q);
      }
      std::vector<int4> sorted;
      sorted.reserve(sitems.size());
      scta_off.assign(P + 1, 0);
      for (int c = 0; c < P; ++c) {
        std::sort(own[c].begin(), own[c].end());  // k-space order within a CTA
        for (int q : own[c]) sorted.push_back(sitems[q]);
        scta_off[c + 1] = (int)sorted.size();
      }
      sitems.swap(sorted);
    }
    p->spread_ctas = P;
  }
  if (blob.empty()) blob.push_back(pad_entry);

  DevAlloc tab{p, &p->table_bytes};
  DevAlloc wrk{p, &p->work_bytes};
  prop_status st;
#define TRY(x)               \
  do {                       \
    st = (x);                \
    if (st != PROP_OK) {     \
      plan_free(p);          \
      return st;             \
    }                        \
  } while (0)
  if (!p->lone_quads) {
    TRY(tab(&p->kb_idx, kb_idx.size(), "sample indices"));
    TRY(tab(&p->kb_w, kb_w.size(), "sample weights"));
    TRY(tab(&p->order, order.size(), "interpolation order"));
  }
  if (!quads.empty()) TRY(tab(&p->quads, quads.size(), "interpolation quads"));
  TRY(tab(&p->phase, phase.size(), "phase table"));
  TRY(tab(&p->deapod, deapod.size(), "deapodisation table"));
  TRY(tab(&p->twiddle, tw.size(), "twiddles"));
  TRY(tab(&p->blade_frame_d, p->blade_frame.size(), "blade frames"));
  const auto cut = [&](InterpCut& c, const std::vector<int4>& items, const std::vector<int>& off) {
    c.n = (int)items.size();
    c.ctas = std::max(1, (int)off.size() - 1);
    if (items.empty()) return PROP_OK;
    const prop_status s = tab(&c.items, items.size(), "interpolation items");
    return s == PROP_OK ? tab(&c.off, off.size(), "interpolation item ranges") : s;
  };
  TRY(cut(p->tile_cut, tile_items, tile_off));
  TRY(cut(p->quad_cut, quad_items, quad_off));
  TRY(tab(&p->sitems, std::max<size_t>(sitems.size(), 1), "spread items"));
  TRY(tab(&p->sitem_cta_off, scta_off.size(), "spread item ranges"));
  TRY(tab(&p->sblob, blob.size(), "spread lists"));
  if (!p->grid_used_h.empty()) TRY(tab(&p->grid_used, p->grid_used_h.size(), "grid block use"));
  TRY(wrk(&p->grid, (size_t)p->T * n * n * p->cs, "grid workspace"));
  TRY(wrk(&p->rows, (size_t)p->T * N * n * p->cs, "row workspace"));
  TRY(wrk(&p->contrib, (size_t)(p->M + 1) * p->cs, "phased residual"));
  // The blocks of the grid that no sample reaches are never written again and
  // hold the zeros that the adjoint columns take them for.  (Before the
  // uploads: those synchronise with it.)
  if (cudaError_t e = cudaMemset(p->grid, 0, (size_t)p->T * n * n * p->cs * sizeof(float2))) {
    plan_free(p);
    return cuda_fail(e, "grid workspace");
  }
  if (!p->lone_quads) {
    TRY(upload(p->kb_idx, kb_idx));
    TRY(upload(p->kb_w, kb_w));
    TRY(upload(p->order, order));
    TRY(upload(p->tile_cut.items, tile_items));
    TRY(upload(p->tile_cut.off, tile_off));
  }
  if (!quads.empty()) {
    TRY(upload(p->quads, quads));
    TRY(upload(p->quad_cut.items, quad_items));
    TRY(upload(p->quad_cut.off, quad_off));
  }
  TRY(upload(p->phase, phase));
  TRY(upload(p->deapod, deapod));
  TRY(upload(p->twiddle, tw));
  TRY(upload(p->blade_frame_d, p->blade_frame));
  if (!sitems.empty()) TRY(upload(p->sitems, sitems));
  TRY(upload(p->sitem_cta_off, scta_off));
  TRY(upload(p->sblob, blob));
  if (p->grid_used) TRY(upload(p->grid_used, p->grid_used_h));
  p->row_kernel = d->row_kernel;
  fft_make_maps(*p);
  if (p->row_kernel == 2 && !p->fused_ws) {
    plan_free(p);
    return fail(PROP_ERR_INVALID_ARG,
                "plan_create: row_kernel 2 needs 2N <= 512, one bin chunk and a bin stride that is a "
                "multiple of 16");
  }
  {
    cudaError_t e = fft_configure(n);
    // The interpolation may use the device's whole opt-in shared memory.
    if (e == cudaSuccess) e = nufft_configure(p->smem_optin);
    if (e != cudaSuccess) {
      plan_free(p);
      return cuda_fail(e, "kernel configuration");
    }
  }
  TRY(tab(&p->status_dev, 1, "status word"));
  if (!alloc && cudaHostAlloc((void**)&p->host_words, 2 * sizeof(double), cudaHostAllocDefault) != cudaSuccess) {
    cudaGetLastError();
    p->host_words = nullptr;  // the calls then copy into pageable memory
  }
  if (p->spread_claimed) TRY(tab(&p->spread_claim, 2, "spread item counter"));
  {
    cudaError_t e = cudaMemset(p->status_dev, 0, sizeof(int));
    if (e == cudaSuccess && p->spread_claim) e = cudaMemset(p->spread_claim, 0, 2 * sizeof(int));
    // the zero row that padding entries of the spread lists point at
    if (e == cudaSuccess) e = cudaMemset(p->contrib + (size_t)p->M * p->cs, 0, (size_t)p->cs * sizeof(float2));
    if (e != cudaSuccess) {
      plan_free(p);
      return cuda_fail(e, "status word");
    }
  }
#undef TRY
  *out = p;
  return PROP_OK;
}

prop_status plan_ensure_recon(Plan* p, int iters) {
  DevAlloc rec{p, &p->recon_bytes};
  prop_status st;
  if (!p->recon_ready) {
    const size_t nv = p->vol_elems();
    const int fused_blocks = (p->Nf + kFftCols - 1) / kFftCols * p->T * p->N;  // fused row kernel's CTAs
    const int red_cap = std::max(1 << 15, fused_blocks);
    if ((st = rec(&p->resid, (size_t)p->M, "residual")) != PROP_OK) return st;
    if ((st = rec(&p->grad, nv, "gradient")) != PROP_OK) return st;
    if ((st = rec(&p->vol2, nv, "volume buffer")) != PROP_OK) return st;
    if ((st = rec(&p->adam_m, nv, "Adam m")) != PROP_OK) return st;
    if ((st = rec(&p->adam_v, nv, "Adam v")) != PROP_OK) return st;
    if ((st = rec(&p->scalars, 8, "loss scalars")) != PROP_OK) return st;
    if ((st = rec(&p->red_interp.partials, red_cap, "partials")) != PROP_OK) return st;
    if ((st = rec(&p->red_interp.counter, 1, "counter")) != PROP_OK) return st;
    if ((st = rec(&p->red_tv.partials, red_cap, "partials")) != PROP_OK) return st;
    if ((st = rec(&p->red_tv.counter, 1, "counter")) != PROP_OK) return st;
    p->red_interp.capacity = red_cap;
    p->red_tv.capacity = red_cap;
    PROP_CUDA(cudaMemset(p->red_interp.counter, 0, sizeof(unsigned int)));
    PROP_CUDA(cudaMemset(p->red_tv.counter, 0, sizeof(unsigned int)));
    p->recon_ready = true;
  }
  if (iters > p->loss_cap) {
    if (p->loss_dev) {
      plan_dev_free(p, p->loss_dev);
      p->recon_bytes -= (size_t)p->loss_cap * sizeof(double);
      p->loss_dev = nullptr;
      p->loss_cap = 0;
    }
    const int cap = std::max(iters, 64);
    if ((st = rec(&p->loss_dev, cap, "loss trace")) != PROP_OK) return st;
    p->loss_cap = cap;
  }
  return PROP_OK;
}

}  // namespace prop

namespace prop {

size_t plan_estimate_bytes(const prop_plan_desc* d, int iters) {
  if (!d || d->n < 8 || d->nf < 1 || d->nblades < 1 || d->lines < 1 || d->readout < 1 || d->nframes < 1)
    return 0;
  const size_t N = d->n, n = 2 * N, Nf = d->nf, B = d->nblades, T = d->nframes;
  const size_t M = B * (size_t)d->lines * d->readout;
  const size_t W = d->kb_width == 8 ? 8 : 6;
  const size_t chunk = d->bin_chunk == 0 ? std::min<size_t>(Nf, kMaxChunk) : std::min<size_t>(d->bin_chunk, Nf);
  const size_t cs = chunk + (chunk & 1);
  const size_t TR = (size_t)interp_tile_rows((int)cs, (int)W), TC = (size_t)interp_tile_cols((int)cs);
  const size_t nquads = B * (((size_t)d->lines + 1) / 2) * (((size_t)d->readout + 1) / 2);
  const size_t ncell = T * n * n;
  const size_t vol = T * N * N * Nf;
  const size_t quads = quad_stride((int)cs) ? nquads : 0;  // the plan may take these, tiles or both
  const size_t interp_items = quads + M / kInterpItem + T * ((n + TR - 1) / TR) * (n / TC) + 1;
  const size_t spread_items = (M * W * W + kSpreadCellCost * ncell) / kSpreadItemCost + 1;
  size_t b = 0;
  b += quads * quad_record((int)W) * 16 + 8 * M + M * (W / 2) * 16;                             // sample tables
  b += (size_t)d->readout * Nf * 8 + 4 * N + 8 * n + 4 * B;
  const size_t cell_lists = 8 * (ncell + spread_items) + 8 * (M * W * W + (kSpreadListPad - 1) * std::min(ncell, M * W * W));
  const size_t group_lists = 8 * (ncell / 4) + 8 + (4 + 16) * 2 * 16 * M + 16 * (ncell / 4);  // items <= groups
  b += 16 * interp_items + 16 * spread_items + std::max(cell_lists, group_lists) + 4 * 1024;  // lists
  b += 8 * T * (n / 2);                                                                             // grid block use
  b += 8 * T * n * n * cs + 8 * T * N * n * cs + 8 * (M + 1) * cs;                                  // workspace
  b += 8 * M + 4 * 8 * vol + 64 + 2 * 8 * std::max<size_t>(std::max<size_t>(32768, interp_items), (Nf + 15) / 16 * T * N) + 8 +
       8 * std::max<size_t>((size_t)std::max(iters, 1), 64);                                           // optimiser
  b += 32 * 512;  // allocation rounding
  return b;
}

}  // namespace prop
