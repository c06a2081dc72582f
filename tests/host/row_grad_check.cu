// Host check, without a GPU, of the rule that takes the fused gradient row kernel
// or the separate passes (fused_rows_grad_pays): plans that measured clearly
// faster one way or the other on a device of 152 SMs, and every plan it takes
// has a kernel.  Prints OK and exits 0 on success.
#include "prop_internal.cuh"
#include <cstdio>
#include <initializer_list>
using namespace prop;
extern int g_fake_registers;  // (fake_runtime.cpp)

static bool fused(int N, int Nf, int T, int chunk = 64) {
  Plan p;
  p.N = N, p.n = 2 * N, p.Nf = Nf, p.T = T, p.num_sms = 152;
  p.chunk = chunk < Nf ? chunk : Nf;
  p.nchunks = (Nf + p.chunk - 1) / p.chunk;
  return fused_rows_grad_pays(p);
}

int main() {
  int fails = g_fake_registers != 64;
#define CHECK(c) do { if (!(c)) ++fails, printf("line %d: %s\n", __LINE__, #c); } while (0)
  CHECK(fused(64, 8, 1) && fused(96, 5, 3) && fused(256, 32, 1) && fused(128, 33, 1) && fused(24, 5, 1));
  CHECK(fused(192, 16, 32) && fused(256, 16, 32) && fused(384, 64, 1) && fused(96, 31, 16) && fused(256, 12, 8));
  CHECK(fused(32, 12, 8) && fused(384, 22, 8));
  CHECK(!fused(512, 1, 32) && !fused(384, 1, 4) && !fused(256, 1, 8) && !fused(192, 5, 32) && !fused(384, 2, 1));
  CHECK(!fused(128, 2, 32) && !fused(16, 64, 32) && !fused(24, 33, 16) && !fused(32, 17, 16) && !fused(32, 2, 8));
  CHECK(!fused(512, 64, 1) && !fused(512, 24, 1, 16) && !fused(64, 64, 1, 32));
  for (int n : {16, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024})
    for (int Nf : {1, 15, 16, 64})
      for (int T : {1, 2, 32}) CHECK(!fused(n / 2, Nf, T) || (n >= 48 && n <= 768));
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails != 0;
}
