// Fused smoothed-TV gradient + Adam update, the TV/loss reduction, and the
// spectral-sum render.
//
// Sec. 4.3 optimises the volume with Adam on the data term plus total
// variation in space and (for dynamic series) time.  Per complex voxel V(x):
//   TV terms sqrt(|d|^2 + eps^2) over forward differences d along x1, x2 and
//   t (no wrap-around); the gradient of one term with respect to its upper
//   end is d / sqrt(|d|^2 + eps^2) and minus that for its lower end;
//   g = gscale * A^H r + tv_xy grad TV_xy + tv_t grad TV_t;
//   per real component: m = b1 m + (1 - b1) g, v = b2 v + (1 - b2) g^2,
//   V -= (lr / (1 - b1^k)) m / (sqrt(v) / sqrt(1 - b2^k) + eps).
// The update reads Vin and writes Vout (ping-pong), because neighbours of a
// voxel are read by other threads.  Bins are fastest, so warps read and write
// contiguous runs; a thread walks a few voxels of one bin along x1.
#include "prop_internal.cuh"
#include "tv_adam.cuh"

namespace prop {
namespace {

constexpr int kOptThreads = 256;
constexpr int kOptLen = 8;   // most voxels that a thread walks

__device__ double block_sum_d(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sh[w] = v;
  __syncthreads();
  const int nw = blockDim.x >> 5;
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = threadIdx.x < nw ? sh[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  __syncthreads();
  return t;
}

struct OptArgs {
  const float2* Vin;
  const float2* g;
  float2* m;
  float2* v;
  float2* out;  // Vout (Adam) or grad (gradient only)
  double* partials;
  unsigned int* counter;
  const double* data_loss;
  double* loss_out;
  int N, Nf, T;
  int fw, nfg, runs, len, nxb;  // a unit: fw bins (of nfg groups) x runs walks of len voxels (of nxb blocks) of a row
  AdamArgs p;
};

// The TV gradient and the update of plans with several bin chunks.  Bound by
// instruction issue, not by its bytes: a flat voxel index with a branch for
// each neighbour took 80 us for the gradient of 512^2 x 24 voxels, whose
// volume, data gradient and result are 151 MB (23 us).  A thread walks kOptLen
// voxels along x1, so that the TV term towards the next voxel is handed on to
// it, a voxel is one offset into each array, every neighbour load is
// unconditional (a missing neighbour reads the voxel itself and is not used)
// and the loads of U voxels are issued together: 55 us (61 us with a 64-bit
// pointer for each row, 64 us at U = 1; U = 4 takes 54 us but 93 registers
// and more).  TT: the volume has time neighbours.  Off: uint32_t while three
// frames are within 4 GB, else size_t.
template <bool ADAM, bool TT, typename Off>
__global__ void __launch_bounds__(kOptThreads) opt_kernel(OptArgs a) {
  grid_dep_wait();
  grid_dep_release();
  constexpr int U = 2;
  const float eps2 = a.p.tv_eps * a.p.tv_eps;
  const bool xy = a.p.tv_xy != 0.f;
  const size_t st = (size_t)a.N * a.N * a.Nf;
  const Off sx = (Off)a.Nf * 8, d2 = (Off)a.N * sx, dt = (Off)st * 8;
  const int run = threadIdx.x / a.fw, fl = threadIdx.x - run * a.fw, per_row = a.nfg * a.nxb;
  const long units = (long)a.T * a.N * per_row;
  float local = 0.f;
  for (long unit = blockIdx.x; unit < units; unit += gridDim.x) {
    const int row = (int)(unit / per_row), rest = (int)(unit - (long)row * per_row);
    const int xb = rest / a.nfg, f = (rest - xb * a.nfg) * a.fw + fl;
    const int i2 = row % a.N, t = row / a.N;
    const int lo = (xb * a.runs + run) * a.len, hi = min(a.N, lo + a.len);
    if (run >= a.runs || f >= a.Nf || lo >= hi) continue;
    const bool h2p = xy && i2 + 1 < a.N, h2m = xy && i2 > 0;
    const bool htp = TT && t + 1 < a.T, htm = TT && t > 0;
    // offsets count from the frame before this one (from this one when t = 0)
    const size_t first = (size_t)(t > 0 ? t - 1 : 0) * st;
    const char* V = reinterpret_cast<const char*>(a.Vin + first);
    char* G = reinterpret_cast<char*>(const_cast<float2*>(a.g) + first);
    char* M1 = reinterpret_cast<char*>(a.m + (ADAM ? first : 0));
    char* M2 = reinterpret_cast<char*>(a.v + (ADAM ? first : 0));
    char* O = reinterpret_cast<char*>(a.out + first);  // may be G
    auto at = [](const char* b, Off o) { return __ldg(reinterpret_cast<const float2*>(b + o)); };
    auto ref = [](char* b, Off o) -> float2& { return *reinterpret_cast<float2*>(b + o); };
    const Off d2p = h2p ? d2 : 0, d2m = h2m ? d2 : 0, dtp = htp ? dt : 0, dtm = htm ? dt : 0;
    Off off = (t > 0 ? dt : 0) + (Off)i2 * d2 + (Off)lo * sx + (Off)f * 8;
    float2 x = at(V, off);
    float mag;
    float2 t1m = make_float2(0.f, 0.f);
    if (xy && lo > 0) t1m = tv_term(csub_rn(x, at(V, off - sx)), eps2, &mag);
    for (int i0 = lo; i0 < hi; i0 += U, off += U * sx) {
      float2 xp[U], x2p[U], x2m[U], xtp[U], xtm[U], gd[U], mm[U], vv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i1 = min(i0 + u, hi - 1);
        const Off c = off + (Off)(i1 - i0) * sx;
        xp[u] = at(V, i1 + 1 < a.N ? c + sx : c);
        x2p[u] = at(V, c + d2p);
        x2m[u] = at(V, c - d2m);
        if constexpr (TT) {
          xtp[u] = at(V, c + dtp);
          xtm[u] = at(V, c - dtm);
        }
        gd[u] = ref(G, c);
        if constexpr (ADAM) {
          mm[u] = ref(M1, c);
          vv[u] = ref(M2, c);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i1 = i0 + u;
        if (i1 >= hi) break;
        const Off c = off + (Off)u * sx;
        // voxel_tv_nb's terms in its order
        float2 gxy = make_float2(0.f, 0.f), gt = make_float2(0.f, 0.f), t1p = make_float2(0.f, 0.f);
        float sxy = 0.f, stt = 0.f;
        if (xy) {
          if (i1 + 1 < a.N) {
            t1p = tv_term(csub_rn(xp[u], x), eps2, &mag);
            gxy = csub_rn(gxy, t1p);
            sxy = __fadd_rn(sxy, mag);
          }
          if (i1 > 0) gxy = cadd_rn(gxy, t1m);
          if (h2p) {
            gxy = csub_rn(gxy, tv_term(csub_rn(x2p[u], x), eps2, &mag));
            sxy = __fadd_rn(sxy, mag);
          }
          if (h2m) gxy = cadd_rn(gxy, tv_term(csub_rn(x, x2m[u]), eps2, &mag));
        }
        if constexpr (TT) {
          if (htp) {
            gt = csub_rn(gt, tv_term(csub_rn(xtp[u], x), eps2, &mag));
            stt = __fadd_rn(stt, mag);
          }
          if (htm) gt = cadd_rn(gt, tv_term(csub_rn(x, xtm[u]), eps2, &mag));
        }
        local = __fadd_rn(local, fmaf(a.p.tv_xy, sxy, __fmul_rn(TT ? a.p.tv_t : 0.f, stt)));
        const float2 g = total_grad(gd[u], gxy, gt, a.p);
        if constexpr (ADAM) {
          const float2 nx = adam_voxel(x, g, mm[u], vv[u], a.p);
          ref(M1, c) = mm[u];
          ref(M2, c) = vv[u];
          ref(O, c) = nx;
        } else {
          ref(O, c) = g;
        }
        t1m = t1p;
        x = xp[u];
      }
    }
  }
  if (a.partials) finish_loss(local, a.partials, a.counter, a.data_loss, a.loss_out);
}

__global__ void render_kernel(const float2* V, float2* img, long npix, int Nf, int lo, int hi) {
  for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < npix; p += (long)gridDim.x * blockDim.x) {
    const float2* v = V + p * Nf;
    float2 s = make_float2(0.f, 0.f);
    for (int f = lo; f < hi; ++f) {
      const float2 x = v[f];
      s.x += x.x;
      s.y += x.y;
    }
    img[p] = s;
  }
}

// PSNR partials: each block writes (sum (|a| - |b|)^2, max |b|^2) of its
// grid-stride share; the last block to arrive combines them in block order
// and writes 10 log10(peak^2 / mse).
__global__ void __launch_bounds__(kOptThreads) psnr_kernel(const float2* a, const float2* b, long count,
                                                           double* scratch, int cap, double* out) {
  double se = 0.0, pk = 0.0;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long)gridDim.x * blockDim.x) {
    const float2 x = a[i], r = b[i];
    const double ma = sqrt((double)x.x * x.x + (double)x.y * x.y);
    const double mr2 = (double)r.x * r.x + (double)r.y * r.y;
    const double d = ma - sqrt(mr2);
    se += d * d;
    pk = fmax(pk, mr2);
  }
  __shared__ double sh[32];
  __shared__ bool last;
  se = block_sum_d(se, sh);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pk = fmax(pk, __shfl_xor_sync(0xffffffffu, pk, o));
  __shared__ double shm[32];
  if ((threadIdx.x & 31) == 0) shm[threadIdx.x >> 5] = pk;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, shm[w]);
    scratch[2 * blockIdx.x] = se;
    scratch[2 * blockIdx.x + 1] = m;
    __threadfence();
    unsigned int* counter = reinterpret_cast<unsigned int*>(scratch + 2 * cap);
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    __threadfence();
    double s = 0.0, m = 0.0;
    for (int i = 0; i < (int)gridDim.x; ++i) {
      s += __ldcg(&scratch[2 * i]);
      m = fmax(m, __ldcg(&scratch[2 * i + 1]));
    }
    const double mse = s / (double)count;
    *out = mse > 0.0 ? 10.0 * log10(m / mse) : __longlong_as_double(0x7ff0000000000000LL);
    *reinterpret_cast<unsigned int*>(scratch + 2 * cap) = 0u;
  }
}

OptArgs make_args(const Plan& p, const float2* Vin, const float2* g, float2* out, const AdamArgs& aa,
                  const Reducer* red, const double* data_loss, double* loss_out) {
  OptArgs a{};
  a.Vin = Vin;
  a.g = g;
  a.out = out;
  a.partials = red ? red->partials : nullptr;
  a.counter = red ? red->counter : nullptr;
  a.data_loss = data_loss;
  a.loss_out = loss_out;
  a.N = p.N;
  a.Nf = p.Nf;
  a.T = p.T;
  const WalkShape w = walk_shape(p.Nf, p.N, kOptThreads, kOptLen);
  a.fw = w.fw;
  a.nfg = w.nfg;
  a.runs = w.runs;
  a.len = w.len;
  a.nxb = w.nxb;
  a.p = aa;
  return a;
}

template <bool ADAM>
cudaError_t launch_opt(const OptArgs& a, bool small, const Reducer* red, cudaStream_t s) {
  const long units = (long)a.T * a.N * a.nfg * a.nxb;
  const long cap = red ? std::min<long>(red->capacity, 16384) : 16384;
  const dim3 grid((unsigned)std::max<long>(1, std::min(units, cap)));
  auto go = [&](auto kern) { return launch_dep(kern, grid, dim3(kOptThreads), 0, s, a); };
  if (a.T > 1 && a.p.tv_t != 0.f)
    return small ? go(opt_kernel<ADAM, true, uint32_t>) : go(opt_kernel<ADAM, true, size_t>);
  return small ? go(opt_kernel<ADAM, false, uint32_t>) : go(opt_kernel<ADAM, false, size_t>);
}

}  // namespace

cudaError_t tv_adam(const Plan& p, const float2* Vin, const float2* g, float2* m, float2* v, float2* Vout,
                    const AdamArgs& aa, const Reducer* red, const double* data_loss, double* loss_out,
                    cudaStream_t s) {
  OptArgs a = make_args(p, Vin, g, Vout, aa, red, data_loss, loss_out);
  a.m = m;
  a.v = v;
  return launch_opt<true>(a, frames_in_32_bits(p), red, s);
}

cudaError_t tv_grad(const Plan& p, const float2* V, const float2* g, float2* grad, const AdamArgs& aa,
                    const Reducer* red, const double* data_loss, double* loss_out, cudaStream_t s) {
  return launch_opt<false>(make_args(p, V, g, grad, aa, red, data_loss, loss_out), frames_in_32_bits(p), red, s);
}

cudaError_t psnr(const Plan& p, const float2* img, const float2* ref, long count, double* out, cudaStream_t s) {
  const unsigned blocks = (unsigned)std::max<long>(1, std::min<long>((count + kOptThreads - 1) / kOptThreads,
                                                                     (long)p.psnr_cap));
  psnr_kernel<<<blocks, kOptThreads, 0, s>>>(img, ref, count, p.psnr_scratch, p.psnr_cap, out);
  return cudaGetLastError();
}

cudaError_t render(const Plan& p, const float2* V, int f_lo, int f_hi, float2* img, cudaStream_t s) {
  const long npix = (long)p.T * p.N * p.N;
  const unsigned blocks = (unsigned)std::min<long>((npix + 255) / 256, 16384);
  render_kernel<<<blocks, 256, 0, s>>>(V, img, npix, p.Nf, f_lo, f_hi);
  return cudaGetLastError();
}

}  // namespace prop

// ---------------------------------------------------------------------------
// Allocation-free TV value and gradient: prop_tv_grad_static.
//
// For callers that cannot allocate device memory (code running inside a
// memory pool or arena owned by a host framework, under a no-allocation
// rule in a real-time loop, or in a callback that must not re-enter the CUDA
// allocator).  It computes the same smoothed TV terms as the optimiser
// kernel, one CTA per image row, and keeps its reduction scratch (one FP64
// partial per image row plus the arrival counter) in the file-scope device
// array below instead of a plan.  The array is 128 KiB + 256 B and stays
// resident on every device that loads the library until the process exits.
#include <mutex>

namespace prop {
namespace {

constexpr int kStaticRows = 16384;       // most image rows (frames * N) per call
constexpr int kStaticDevices = 64;

// [0, kStaticRows): per-row partial sums; slot kStaticRows holds the counter.
static __device__ __align__(256) double g_tv_static_scratch[kStaticRows + 32];

__global__ void __launch_bounds__(kOptThreads)
tv_grad_rows_kernel(const float2* V, float2* grad, double* scratch, double* loss_out, int N, int Nf, int T,
                    float tv_xy, float tv_t, float tv_eps) {
  const float eps2 = tv_eps * tv_eps;
  const int rowlen = N * Nf;
  const int row = blockIdx.x;  // t * N + i2
  const int i2 = row % N;
  const int t = row / N;
  const long rbase = (long)row * rowlen;
  float local = 0.f;
  for (int e = threadIdx.x; e < rowlen; e += blockDim.x) {
    const long idx = rbase + e;
    const float2 x = V[idx];
    float2 gxy, gt;
    local += voxel_tv(V, (size_t)idx, x, e / Nf, i2, t, N, Nf, T, tv_xy, tv_t, eps2, &gxy, &gt);
    grad[idx] = make_float2(fmaf(tv_xy, gxy.x, tv_t * gt.x), fmaf(tv_xy, gxy.y, tv_t * gt.y));
  }
  __shared__ double sh[32];
  __shared__ bool last;
  unsigned int* counter = reinterpret_cast<unsigned int*>(scratch + kStaticRows);
  const double bs = block_sum_d((double)local, sh);
  if (threadIdx.x == 0) {
    scratch[row] = bs;
    __threadfence();
    const unsigned prev = atomicAdd(counter, 1u);
    last = prev == gridDim.x - 1;
  }
  __syncthreads();
  if (last) {
    __threadfence();
    double s = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) s += __ldcg(&scratch[i]);
    s = block_sum_d(s, sh);
    if (threadIdx.x == 0) {
      *loss_out = s;
      *counter = 0u;
    }
  }
}

std::mutex g_static_mutex;
double* g_static_addr[kStaticDevices] = {};

}  // namespace
}  // namespace prop

extern "C" prop_status prop_tv_grad_static(const void* V_dev, int nframes, int n, int nf, float tv_xy,
                                           float tv_t, float tv_eps, void* grad_dev, double* loss_dev,
                                           void* stream) {
  using namespace prop;
  if (!V_dev || !grad_dev || !loss_dev) return fail(PROP_ERR_INVALID_ARG, "tv_grad_static: null argument");
  if (((uintptr_t)V_dev & 15u) || ((uintptr_t)grad_dev & 15u) || ((uintptr_t)loss_dev & 7u))
    return fail(PROP_ERR_INVALID_ARG, "tv_grad_static: V and grad must be 16-byte aligned, loss 8-byte aligned");
  if (V_dev == grad_dev) return fail(PROP_ERR_INVALID_ARG, "tv_grad_static: V and grad must not alias");
  if (nframes < 1 || n < 1 || nf < 1 || (long long)n * nf > (1LL << 30))
    return fail(PROP_ERR_INVALID_ARG, "tv_grad_static: nframes, n, nf must be >= 1 and n * nf <= 2^30");
  if ((long long)nframes * n > kStaticRows)
    return fail(PROP_ERR_INVALID_ARG, "tv_grad_static: nframes * n = " + std::to_string((long long)nframes * n) +
                                          " image rows exceeds the static scratch limit of " +
                                          std::to_string(kStaticRows));
  if (!(tv_eps > 0.f) || !(tv_xy >= 0.f) || !(tv_t >= 0.f))
    return fail(PROP_ERR_INVALID_ARG, "tv_grad_static: need tv_xy >= 0, tv_t >= 0, tv_eps > 0");
  int dev = 0;
  PROP_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kStaticDevices) return fail(PROP_ERR_INVALID_ARG, "tv_grad_static: device ordinal too large");
  double* scratch = nullptr;
  {
    // One-time set-up per device, with that device current: the host-side
    // name of the array is not a device address, so look the address up.
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_addr[dev]) {
      void* addr = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&addr, g_tv_static_scratch);
      if (e != cudaSuccess) return cuda_fail(e, "tv_grad_static: cudaGetSymbolAddress");
      g_static_addr[dev] = static_cast<double*>(addr);
    }
    scratch = g_static_addr[dev];
  }
  cudaStream_t s = (cudaStream_t)stream;
  // The counter must start at zero; the partials are fully rewritten each call.
  PROP_CUDA(cudaMemsetAsync(scratch + kStaticRows, 0, sizeof(double), s));
  tv_grad_rows_kernel<<<nframes * n, kOptThreads, 0, s>>>((const float2*)V_dev, (float2*)grad_dev, scratch,
                                                           loss_dev, n, nf, nframes, tv_xy, tv_t, tv_eps);
  PROP_CUDA(cudaGetLastError());
  return PROP_OK;
}
