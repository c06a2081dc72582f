// Host check, without a GPU, of what a plan does when the warp-specialised row
// kernel was compiled for fewer registers than its two groups share out: the
// transforms of its length still configure, and the plan takes the per-row
// kernel.  The runtime calls involved are replaced by fakes that report a
// register count (fake_runtime.cpp).  Prints OK and exits 0 on success.
#include "prop_internal.cuh"
#include <cstdio>

extern int g_fake_registers;

int main() {
  using namespace prop;
  int fails = 0;
  for (int n : {128, 384, 512})
    for (int regs : {64, 56}) {
      g_fake_registers = regs;
      if (fft_configure(n) != cudaSuccess) ++fails, printf("2N = %d at %d registers: refused\n", n, regs);
      for (int row_kernel : {0, 1, 2}) {
        Plan p;
        p.n = n, p.N = n / 2, p.Nf = p.cs = p.chunk = 16, p.nchunks = 1, p.T = 32, p.num_sms = 152;
        p.smem_optin = 227 * 1024;
        p.row_kernel = row_kernel;
        fft_make_maps(p);
        const bool split = n >= 384;  // the two groups are of one size
        if (p.fused_ws != (row_kernel != 1 && (!split || regs >= 64)))
          ++fails, printf("2N = %d at %d registers, row kernel %d: %d\n", n, regs, row_kernel, p.fused_ws);
      }
    }
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails != 0;
}
