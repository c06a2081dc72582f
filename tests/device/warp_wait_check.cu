// Check of mbar_wait_warp (tma.cuh) on a GPU: eight warps wait on a barrier
// that never completes, every lane with a limit of its own (20 to 640 us of SM
// clock), so that the lanes of a warp leave the wait at different times while
// other warps set the flag.  The decision has to be one per warp, at every
// wait, and the shuffles that follow it have to find the whole warp.  Prints OK
// and exits 0 on success.
#include "tma.cuh"
#include <cstdio>

using namespace prop;

constexpr int kWarps = 8, kRounds = 4;

__global__ void __launch_bounds__(32 * kWarps) check(int* went_on, int* sums, int open_round) {
  __shared__ uint64_t bar[kRounds];
  __shared__ volatile int abort;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int r = 0; r < kRounds; ++r) mbar_init(&bar[r], 1);
    fence_mbar_init();
    abort = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int r = 0; r < open_round; ++r) mbar_arrive(&bar[r]);  // the others never complete
  for (int r = 0; r < kRounds; ++r) {
    const bool on = mbar_wait_warp(&bar[r], 0, &abort, 40000LL * (1 + (lane * 7 + warp * 13) % 32));
    went_on[(r * kWarps + warp) * 32 + lane] = on ? 1 : 0;
    if (!on) break;
    int v = 1;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    sums[(r * kWarps + warp) * 32 + lane] = v;
  }
}

int main() {
  const int n = kRounds * kWarps * 32;
  int *d = nullptr, h[2 * n], fails = 0;
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return 2;
  for (int open = 0; open <= kRounds; ++open)
    for (int rep = 0; rep < 20; ++rep) {
      cudaMemset(d, 0xff, sizeof(h));
      check<<<1, 32 * kWarps>>>(d, d + n, open);
      if (cudaDeviceSynchronize() != cudaSuccess || cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess)
        return 3;
      for (int w = 0; w < kWarps; ++w)
        for (int r = 0; r < kRounds; ++r)
          for (int l = 0; l < 32; ++l) {
            const int i = (r * kWarps + w) * 32 + l;
            fails += h[i] != h[(r * kWarps + w) * 32];     // one decision a warp
            fails += h[i] == 1 && h[n + i] != 32;          // and the whole warp in what follows
            fails += r >= open && h[i] == 1;               // an open barrier is never passed
            fails += open == kRounds && h[i] != 1;         // nobody gives up where all complete
          }
    }
  cudaFree(d);
  printf(fails ? "FAIL %d\n" : "OK\n", fails);
  return fails != 0;
}
