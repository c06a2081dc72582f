// Prints the number of spread items that a plan of the given geometry lists
// (grouped lists) and the least number from which the CTAs of a device with the
// given count of SMs claim them at run time: the list builder on the host, no
// GPU.  Arguments: N, bins, blades, lines, readout, width, SMs; blade b at angle
// pi b / blades, one frame.
#include "plan.cu"
#include <cstdio>
#include <cstdlib>
using namespace prop;

int main(int argc, char** argv) {
  if (argc != 8) return 2;
  const int N = atoi(argv[1]), Nf = atoi(argv[2]), B = atoi(argv[3]), L = atoi(argv[4]), R = atoi(argv[5]);
  const int W = atoi(argv[6]), sms = atoi(argv[7]);
  Plan p;
  p.N = N, p.n = 2 * N, p.W = W, p.cs = Nf + (Nf & 1), p.T = 1, p.B = B, p.L = L, p.R = R, p.M = B * L * R;
  p.blade_frame.assign(B, 0);
  std::vector<int> tap;
  for (int b = 0; b < B; ++b)
    for (int l = 0; l < L; ++l)
      for (int j = 0; j < R; ++j) {
        const double th = std::acos(-1.0) * b / B, kp = (l - L / 2.0) / N, kr = (j - R / 2.0) / N;
        const double k[2] = {kr * std::cos(th) - kp * std::sin(th), kr * std::sin(th) + kp * std::cos(th)};
        for (int a = 0; a < 2; ++a) {
          double u = p.n * k[a];
          u -= p.n * std::floor(u / p.n);
          tap.push_back(((int)std::floor(u) - (W / 2 - 1) + p.n) % p.n);
        }
      }
  const std::vector<double> wd((size_t)p.M * 2 * W, 1.0);
  std::vector<int4> items;
  std::vector<int2> blob;
  mark_used_blocks(p, tap);
  if (!build_group_lists(p, tap, wd, items, blob)) return 3;
  printf("%zu %d\n", items.size(), kSpreadClaimMinItems * kSpreadCtasPerSm * sms);
  return 0;
}
