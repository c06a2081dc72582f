// Batched shared-memory FFTs of the oversampled grid (no cuFFT).
//
// The 2N x 2N transform of every (frame, bin) slice is done as two passes of
// 1-D transforms of length n = 2N along one axis, each CTA transforming a
// tile of kFftCols = 16 lines (8 in the long row passes) that are adjacent in
// memory, so that every global access of a warp covers two runs of 16
// consecutive complex64 values (2 x 128 B, fully coalesced).  Bins are the fastest axis of every
// array, so the "lines" of a pass are (u1, f) columns of the grid or the
// bins of one image row.
//
// Each 1-D transform is a mixed-radix Stockham FFT (radix_plan):
// pass p with radix R and stride Ns (product of the previous radices)
// reads R values at stride n/R, multiplies by exp(-+2 pi i r (j mod Ns) /
// (Ns R)), does an R-point DFT in registers and writes the results at
// (j / Ns) Ns R + (j mod Ns) + r Ns.  The first pass reads global memory
// directly (zero padding and deapodisation applied on the fly), the last
// pass writes global memory directly (cropping and scaling applied on the
// fly); intermediate passes exchange through shared memory in place.
// Every thread holds E = 16 (n = 2^a) or 12 (n = 3 * 2^a) values per pass,
// 32 and 24 in the long transforms (kValsPlain, kValsCols).
#include <type_traits>

#include "prop_internal.cuh"
#include "tv_adam.cuh"
#include "tma.cuh"

namespace prop {
namespace {

struct RadixPlan {
  int count;
  int r[8];
};

// Radices for E values a thread (a thread holds whole butterflies in every
// pass): with E = 32, radix 32 while it divides and then 16; with E = 24,
// radix 24 and then the rest (16 or 32) in one pass, of which some warps take
// a butterfly more than others; else every radix divides E, radix 8 where E
// allows (E = 16), radix 4 where it does not (E = 12, lengths with a factor 3:
// half the registers of 24, twice the threads); then 4, 2 and the threes, a
// leftover factor 2 merged with a 3 into one radix-6 pass.
__host__ __device__ constexpr RadixPlan radix_plan(int n, int E) {
  RadixPlan p{0, {1, 1, 1, 1, 1, 1, 1, 1}};
  int m = n, threes = 0;
  while (m % 3 == 0) {
    m /= 3;
    ++threes;
  }
  if (E == 24) {
    p.r[p.count++] = 24;
    p.r[p.count++] = n / 24;
    return p;
  }
  while (E % 32 == 0 && threes == 0 && m % 32 == 0) {
    p.r[p.count++] = 32;
    m /= 32;
  }
  if (E % 16 == 0 && threes == 0 && m % 16 == 0 && p.count > 0) {
    p.r[p.count++] = 16;
    m /= 16;
  }
  while (E % 8 == 0 && m % 8 == 0) {
    p.r[p.count++] = 8;
    m /= 8;
  }
  while (threes > 0 && m % 4 == 0) {
    p.r[p.count++] = 4;
    m /= 4;
  }
  if (m % 4 == 0) {
    p.r[p.count++] = 4;
    m /= 4;
  }
  if (m % 2 == 0 && threes > 0) {  // a leftover 2 and a 3 make one radix-6 pass
    m /= 2;
    --threes;
    for (int i = 0; i < threes; ++i) p.r[p.count++] = 3;
    p.r[p.count++] = 6;
    return p;
  }
  if (m % 2 == 0) {
    p.r[p.count++] = 2;
    m /= 2;
  }
  for (int i = 0; i < threes; ++i) p.r[p.count++] = 3;
  return p;
}

// Twiddle tables, one per Stockham pass p >= 1 with stride NS and radix R:
// entry [k][r] (k < NS, r < R) = exp(-2 pi i r k / (NS R)), so a butterfly
// fetches its R factors with R/2 16-byte loads.  Offsets are even (every NS
// and hence every table size is even), so the tables stay 16-byte aligned.
template <int NFFT, int EV>
__host__ __device__ constexpr int tw_offset(int pass) {
  constexpr RadixPlan RP = radix_plan(NFFT, EV);
  int off = 0, ns = RP.r[0];
  for (int q = 1; q < pass; ++q) {
    off += ns * RP.r[q];
    ns *= RP.r[q];
  }
  return off;
}

// Values per thread of the row passes, alone and fused (the same, so that they
// round alike): 16 (two radix-8 butterflies a pass), 12 for lengths with a
// factor 3 (radices 4, 2, 3); above 512 points, where one CTA of 1024 threads
// was all that fitted an SM, 32 and 24, which make two passes as in the columns
// (768 points, 64 bins: forward 82 -> 64 us, adjoint 72 -> 62, fused update
// 248 -> 229; 1024 points 41 -> 36 and 36 -> 36 us; 32 at 512 points leaves the
// fused update half its threads, 56 -> 68 us).  The image transforms of the
// projection model, 4 lines a CTA, keep 16 and 12.
template <int NFFT>
constexpr int kValsPlain = NFFT == 1024 ? 32 : NFFT == 768 ? 24 : NFFT % 3 == 0 ? 12 : 16;
template <int NFFT>
constexpr int kValsFused = kValsPlain<NFFT>;
template <int NFFT>
constexpr int kValsCart = NFFT % 3 == 0 ? 12 : 16;
// Values per thread of the column passes, as many as make two passes of them
// (one shared-memory exchange): 32 at n = 512 (radix 32 then 16) and 1024 (32,
// 32), 24 at n = 384 (24, 16) and 768 (24, 32), with twice the registers and
// half the threads of a 16- or 12-value shape.  The exchanges and the twiddle
// products between passes are what the passes spend their issue slots and
// shared-memory wavefronts on (60 % of both at 2N = 384).  2N = 512: 23.9 ->
// 20.3 us forward, 24.8 -> 22.3 us adjoint; 384 (64 bins, 16 frames): 126 -> 113
// us and 128 -> 111 us (with radices 8, 8, 6); 768: 142 -> 82 us and 146 -> 84
// us (12 values a thread before, the forward pass spilling); 1024: 98 -> 39 us
// and 62 -> 53 us.
template <int NFFT>
constexpr int kValsCols = NFFT == 512 || NFFT == 1024 ? 32 : NFFT == 384 || NFFT == 768 ? 24 : kValsPlain<NFFT>;

template <int NFFT, int EV>
struct Shape {
  static constexpr int E = EV;                 // values per thread
  static constexpr int TPL = NFFT / E;         // threads per line
  static constexpr int THREADS = TPL * kFftCols;
  static constexpr int TW = tw_offset<NFFT, EV>(radix_plan(NFFT, EV).count);  // twiddle table entries
  static constexpr size_t SMEM = (size_t)NFFT * kFftCols * sizeof(float2) + (size_t)TW * sizeof(float2);
};

// The thread's place in its line (COLS lines side by side); the mask tells the
// compiler its range, so that what depends on a position's block or on the
// crop is decided at compile time where TPL divides it.
template <int NFFT, int EV, int COLS = kFftCols>
__device__ __forceinline__ int line_thread(int tid) {
  constexpr int TPL = Shape<NFFT, EV>::TPL;
  static_assert((TPL & (TPL - 1)) == 0, "threads a line: a power of two");
  return (tid / COLS) & (TPL - 1);
}

// Fill the per-pass twiddle tables from the length-NFFT table exp(-2 pi i m / NFFT).
template <int NFFT, int EV>
__device__ void build_twiddles(float2* tws, const float2* __restrict__ base) {
  constexpr RadixPlan RP = radix_plan(NFFT, EV);
  int ns = RP.r[0];
  for (int p = 1; p < RP.count; ++p) {
    const int R = RP.r[p];
    const int off = tw_offset<NFFT, EV>(p);
    const int step = NFFT / (ns * R);
    for (int idx = threadIdx.x; idx < ns * R; idx += blockDim.x) {
      const int k = idx / R, r = idx - (idx / R) * R;
      tws[off + idx] = base[r * k * step];
    }
    ns *= R;
  }
}

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// Rounded product that is never contracted into a later add: the inputs of
// the first butterfly round the same way in every kernel that builds them.
__device__ __forceinline__ float2 cscale_rn(float2 a, float s) {
  return make_float2(__fmul_rn(a.x, s), __fmul_rn(a.y, s));
}
// z * (SIGN i)
template <int SIGN>
__device__ __forceinline__ float2 mul_si(float2 z) {
  return SIGN > 0 ? make_float2(-z.y, z.x) : make_float2(z.y, -z.x);
}

// In-register DFTs X_k = sum_q v_q exp(SIGN 2 pi i q k / R).
template <int R, int SIGN>
struct Dft;

template <int SIGN>
struct Dft<2, SIGN> {
  __device__ __forceinline__ static void run(float2* v) {
    float2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};

template <int SIGN>
struct Dft<4, SIGN> {
  __device__ __forceinline__ static void run(float2* v) {
    float2 t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
    float2 t2 = cadd(v[1], v[3]), t3 = mul_si<SIGN>(csub(v[1], v[3]));
    v[0] = cadd(t0, t2);
    v[2] = csub(t0, t2);
    v[1] = cadd(t1, t3);
    v[3] = csub(t1, t3);
  }
};

template <int SIGN>
struct Dft<8, SIGN> {
  __device__ __forceinline__ static void run(float2* v) {
    constexpr float h = 0.70710678118654752f;  // 1/sqrt(2)
    float2 a[4], b[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      a[q] = cadd(v[q], v[q + 4]);
      b[q] = csub(v[q], v[q + 4]);
    }
    // b_q *= w^q, w = exp(SIGN i pi / 4)
    {
      float2 z = b[1];
      b[1] = make_float2((z.x - SIGN * z.y) * h, (z.y + SIGN * z.x) * h);
      b[2] = mul_si<SIGN>(b[2]);
      z = b[3];
      b[3] = make_float2((-z.x - SIGN * z.y) * h, (-z.y + SIGN * z.x) * h);
    }
    Dft<4, SIGN>::run(a);
    Dft<4, SIGN>::run(b);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      v[2 * q] = a[q];
      v[2 * q + 1] = b[q];
    }
  }
};

template <int SIGN>
struct Dft<3, SIGN> {
  __device__ __forceinline__ static void run(float2* v) {
    constexpr float s3 = 0.86602540378443865f;  // sqrt(3)/2
    float2 t = cadd(v[1], v[2]);
    float2 m = make_float2(v[0].x - 0.5f * t.x, v[0].y - 0.5f * t.y);
    float2 d = mul_si<SIGN>(cscale(csub(v[1], v[2]), s3));
    v[0] = cadd(v[0], t);
    v[1] = cadd(m, d);
    v[2] = csub(m, d);
  }
};

// 6 = 2 x 3: the three-point DFTs of the even and the odd inputs, then
// X[k] = E[k] + w^k O[k] and X[k + 3] = E[k] - w^k O[k], w = exp(SIGN 2 pi i / 6).
template <int SIGN>
struct Dft<6, SIGN> {
  __device__ __forceinline__ static void run(float2* v) {
    constexpr float s3 = 0.86602540378443865f;  // sqrt(3)/2
    float2 a[3] = {v[0], v[2], v[4]}, b[3] = {v[1], v[3], v[5]};
    Dft<3, SIGN>::run(a);
    Dft<3, SIGN>::run(b);
    const float2 t1 = make_float2(0.5f * b[1].x - SIGN * s3 * b[1].y, 0.5f * b[1].y + SIGN * s3 * b[1].x);
    const float2 t2 = make_float2(-0.5f * b[2].x - SIGN * s3 * b[2].y, -0.5f * b[2].y + SIGN * s3 * b[2].x);
    v[0] = cadd(a[0], b[0]);
    v[3] = csub(a[0], b[0]);
    v[1] = cadd(a[1], t1);
    v[4] = csub(a[1], t1);
    v[2] = cadd(a[2], t2);
    v[5] = csub(a[2], t2);
  }
};

// cos(2 pi m / 32) from its values on the first quadrant; sin(2 pi m / 32)
// = cos(2 pi (m - 8) / 32).  The constant factors inside the radix-16 and
// radix-32 butterflies.
__host__ __device__ constexpr double cos32(int m) {
  constexpr double q[9] = {1.0,
                           0.98078528040323044912618223613424,   // cos(pi / 16)
                           0.92387953251128675612818318939679,   // cos(pi / 8)
                           0.83146961230254523707878837761791,   // cos(3 pi / 16)
                           0.70710678118654752440084436210485,   // cos(pi / 4)
                           0.55557023301960222474283081394853,   // cos(5 pi / 16)
                           0.38268343236508977172845998403040,   // cos(3 pi / 8)
                           0.19509032201612826784828486847702,   // cos(7 pi / 16)
                           0.0};
  m &= 31;
  return m <= 8 ? q[m] : m <= 16 ? -q[16 - m] : m <= 24 ? -q[m - 16] : q[32 - m];
}
__host__ __device__ constexpr double sin32(int m) { return cos32(m - 8); }

// cos(2 pi m / 24) and sin(2 pi m / 24) likewise, for the radix-24 butterfly.
__host__ __device__ constexpr double cos24(int m) {
  constexpr double q[7] = {1.0,
                           0.96592582628906828674974319972890,   // cos(pi / 12)
                           0.86602540378443864676372317075294,   // cos(pi / 6)
                           0.70710678118654752440084436210485,   // cos(pi / 4)
                           0.5,
                           0.25881904510252076234889883762405,   // cos(5 pi / 12)
                           0.0};
  m = (m % 24 + 24) % 24;
  return m <= 6 ? q[m] : m <= 12 ? -q[12 - m] : m <= 18 ? -q[m - 12] : q[24 - m];
}
__host__ __device__ constexpr double sin24(int m) { return cos24(m - 6); }

// z * exp(SIGN 2 pi i M / R) for R dividing 32 or R = 24; quarter turns exactly.
template <int SIGN, int R, int M>
__device__ __forceinline__ float2 rotate(float2 z) {
  constexpr int D = R == 24 ? 24 : 32;
  constexpr int m = (M % R) * (D / R);  // in D-ths of a turn
  if constexpr (m == 0) {
    return z;
  } else if constexpr (4 * m == D) {
    return mul_si<SIGN>(z);
  } else if constexpr (2 * m == D) {
    return make_float2(-z.x, -z.y);
  } else if constexpr (4 * m == 3 * D) {
    return mul_si<-SIGN>(z);
  } else {
    constexpr float c = (float)(D == 24 ? cos24(m) : cos32(m));
    constexpr float sn = (float)(SIGN * (D == 24 ? sin24(m) : sin32(m)));
    return make_float2(fmaf(z.x, c, -z.y * sn), fmaf(z.x, sn, z.y * c));
  }
}

template <int I, int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

// R = R1 R2 point DFT from R2 DFTs of R1 points and R1 of R2 points:
// with q = R2 q1 + q2 and k = k1 + R1 k2,
//   X_k = sum_q2 w_R^(q2 k1) w_R2^(q2 k2) sum_q1 x_q w_R1^(q1 k1),  w_R = exp(SIGN 2 pi i / R).
template <int R1, int R2, int SIGN>
__device__ __forceinline__ void dft_compose(float2* v) {
  constexpr int R = R1 * R2;
  float2 y[R];  // y[q2 R1 + k1]
  static_for<0, R2>([&](auto q2c) {
    constexpr int q2 = decltype(q2c)::value;
    float2 a[R1];
#pragma unroll
    for (int q1 = 0; q1 < R1; ++q1) a[q1] = v[R2 * q1 + q2];
    Dft<R1, SIGN>::run(a);
    static_for<0, R1>([&](auto k1c) {
      constexpr int k1 = decltype(k1c)::value;
      y[q2 * R1 + k1] = rotate<SIGN, R, q2 * k1>(a[k1]);
    });
  });
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) {
    float2 b[R2];
#pragma unroll
    for (int q2 = 0; q2 < R2; ++q2) b[q2] = y[q2 * R1 + k1];
    Dft<R2, SIGN>::run(b);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) v[k1 + R1 * k2] = b[k2];
  }
}

template <int SIGN>
struct Dft<16, SIGN> {
  __device__ __forceinline__ static void run(float2* v) { dft_compose<4, 4, SIGN>(v); }
};
template <int SIGN>
struct Dft<32, SIGN> {
  __device__ __forceinline__ static void run(float2* v) { dft_compose<8, 4, SIGN>(v); }
};

template <int SIGN>
struct Dft<24, SIGN> {
  __device__ __forceinline__ static void run(float2* v) { dft_compose<8, 3, SIGN>(v); }
};

// One Stockham pass; recurses into the next pass at compile time.
// PIN: the input line is a zero-padded image line (image index i at
// position i - N/2 mod n, N = n/2, zeros elsewhere); the first pass then
// reads only the positions that hold image values, known at compile time
// for radix 8 or 4 (r < R/4 or r >= 3R/4), and never touches the padding.
// POUT likewise for a cropped output in the last pass: only the image
// positions are formed and stored.
struct NoHook {
  __device__ void operator()() const {}
};

// Barrier between passes: the whole CTA, or a named barrier over the first
// COUNT threads when only part of the CTA transforms.
struct CtaSync {
  __device__ static void sync() { __syncthreads(); }
};
template <int ID, int COUNT>
struct GroupSync {
  static_assert(COUNT % 32 == 0, "named barriers count whole warps");
  __device__ static void sync() { asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(COUNT) : "memory"); }
};

// `hook` runs once, on every thread, right after the barrier that follows
// the first pass (all reads of the first pass's input are then complete).
// COLS: lines a tile (the stride of the exchange buffer X[pos][col]).
template <int NFFT, int EV, int SIGN, int PI, int NS, bool PIN, bool POUT, class Sync = CtaSync, class In,
          class Out, class Hook = NoHook, int COLS = kFftCols>
__device__ __forceinline__ void fft_pass(float2* X, const float2* tws, int col, int tl, const In& in,
                                         const Out& out, const Hook& hook = Hook()) {
  constexpr RadixPlan RP = radix_plan(NFFT, EV);
  constexpr int R = RP.r[PI];
  constexpr int TPL = NFFT / EV;
  constexpr int STRIDE = NFFT / R;                 // butterflies a line
  constexpr int NB = (STRIDE + TPL - 1) / TPL;     // and a thread
  constexpr bool EVEN = STRIDE % TPL == 0;         // else some warps sit the last one out
  static_assert((STRIDE % TPL) * COLS % 32 == 0, "whole warps");
  // With 8 lines a tile a half-warp's two positions are in different halves of
  // the banks when they are read, and would be in the same half when they are
  // written (R apart): odd rows of the R0 x R1 exchange swap their neighbours.
  constexpr bool SWAP = COLS == 8 && RP.count == 2 && RP.r[0] % 2 == 0;
  constexpr bool FIRST = PI == 0;
  constexpr bool LAST = PI == RP.count - 1;
  constexpr bool PRUNE_IN = FIRST && PIN && R % 4 == 0;
  constexpr bool PRUNE_OUT = LAST && POUT && R % 4 == 0;
  constexpr int Q = NFFT / 4;  // N / 2
  static_assert(!(FIRST && PIN) || PRUNE_IN, "padded input needs a first radix that 4 divides");
  float2 v[NB * R];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int j = tl + TPL * q;
    if (!EVEN && j >= STRIDE) continue;
    const int k = LAST ? j : j % NS;  // (NS R = NFFT in the last pass)
    float2 w[R];
    if constexpr (NS > 1) {
      const float2* T = tws + tw_offset<NFFT, EV>(PI) + k * R;
      if constexpr (R % 2 == 0) {
#pragma unroll
        for (int h = 0; h < R / 2; ++h) {
          const float4 t = reinterpret_cast<const float4*>(T)[h];
          w[2 * h] = make_float2(t.x, t.y);
          w[2 * h + 1] = make_float2(t.z, t.w);
        }
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) w[r] = T[r];
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int pos = j + r * STRIDE;
      float2 x;
      if constexpr (PRUNE_IN) {
        if (r < R / 4)
          x = in.at(pos + Q, col);
        else if (r >= R - R / 4)
          x = in.at(pos - 3 * Q, col);
        else
          x = make_float2(0.f, 0.f);
      } else if constexpr (FIRST) {
        x = in(pos, col);
      } else {
        x = X[(SWAP ? r * STRIDE + (j ^ (r & 1)) : pos) * COLS + col];
      }
      if constexpr (NS > 1) {
        if (r > 0) x = SIGN < 0 ? cmul(x, w[r]) : cmulc(x, w[r]);
      }
      v[q * R + r] = x;
    }
    Dft<R, SIGN>::run(v + q * R);
  }
  if constexpr (!LAST) {
    if constexpr (!FIRST) Sync::sync();  // every read of this pass is done
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int j = tl + TPL * q;
      if (!EVEN && j >= STRIDE) continue;
      const int d = (j / NS) * NS * R + (j % NS);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int pos = SWAP ? d + r + (r & 1 ? -(j & 1) : j & 1) : d + r * NS;
        X[pos * COLS + col] = v[q * R + r];
      }
    }
    Sync::sync();
    if constexpr (FIRST) hook();
    fft_pass<NFFT, EV, SIGN, PI + 1, NS * R, PIN, POUT, Sync, In, Out, Hook, COLS>(X, tws, col, tl, in, out, hook);
  } else {
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int d = tl + TPL * q;  // NS R = NFFT in the last pass, so (j / NS) NS R + j % NS = j
      if (!EVEN && d >= STRIDE) continue;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if constexpr (PRUNE_OUT) {
          if (r < R / 4)
            out.at(d + r * NS + Q, col, v[q * R + r]);
          else if (r >= R - R / 4)
            out.at(d + r * NS - 3 * Q, col, v[q * R + r]);
        } else {
          out(d + r * NS, col, v[q * R + r]);
        }
      }
    }
  }
}

// Position p of a line of length n = 2N holds image index i = x + N/2 for
// x = p (p < N/2) or x = p - n (p >= n - N/2); other positions are padding.
template <int n>
__device__ __forceinline__ int image_index(int p) {
  constexpr int h = n / 4;
  if (p < h) return p + h;
  if (p >= n - h) return p - (n - h);
  return -1;
}

// The value `off` bytes past `base`.  The passes address global memory as a
// base that is the same for the whole CTA plus a 32-bit byte offset (an image
// row of V or of the row intermediate, one frame's grid: all below 4 GB), and
// the lengths n and N are compile-time, so that an access costs one multiply-add
// and the crop is decided at compile time where a thread's positions allow:
// the adjoint column pass at 2N = 384 issued 58 instructions a value with
// run-time lengths and 64-bit indices.
__device__ __forceinline__ float2 load_at(const void* base, uint32_t off) {
  return __ldg(reinterpret_cast<const float2*>(static_cast<const char*>(base) + off));
}
__device__ __forceinline__ void store_at(void* base, uint32_t off, float2 v) {
  *reinterpret_cast<float2*>(static_cast<char*>(base) + off) = v;
}

struct FftArgs {
  const float2* src;
  float2* dst;
  const float* deapod;
  const float2* twiddle;
  int Nf;
  int C;   // bin stride of the workspace (the plan's chunk)
  int Cv;  // valid bins in this chunk (<= C)
  int f0;
  float scale;
  const uint64_t* used;  // column passes: grid blocks in use [frame][u1 / 2], or null
  int ushift;            // log2 of the 16-line tiles in two grid columns
};

// Blocks in use of the grid column that 16-line tile qt of frame t lies in
// (bin strides 8 to 64: two adjacent columns hold a whole number of tiles).
__device__ __forceinline__ uint64_t used_blocks(const uint64_t* used, int ushift, int n, size_t t, int qt) {
  return used ? __ldg(&used[t * (n >> 1) + (qt >> ushift)]) : ~0ull;
}

enum Kind { kFwdRows = 0, kFwdCols = 1, kAdjCols = 2, kAdjRows = 3 };

// Forward rows: V[t][i2][i1][f0 + f] * c(i1) c(i2), padded -> rows[t][i2][u1][f].
struct InFwdRows {
  const float2* V;  // voxel (t, i2, 0, f0 + fbase)
  const float* dp;
  uint32_t step;    // bytes from one voxel of the row to the next
  int live;         // valid bins from fbase on
  float c2;
  __device__ float2 at(int i1, int col) const {  // i1: image index
    if (col >= live) return make_float2(0.f, 0.f);
    return cscale_rn(load_at(V, (uint32_t)i1 * step + (uint32_t)col * 8u), dp[i1] * c2);
  }
};
struct OutFwdRows {
  float2* rows;   // position (row, 0, fbase)
  uint32_t step;  // bytes from one position to the next
  int live;       // bins of the stride from fbase on
  __device__ void operator()(int pos, int col, float2 val) const {
    if (col < live) store_at(rows, (uint32_t)pos * step + (uint32_t)col * 8u, val);
  }
};
// Forward columns: rows[t][i2][q], padded along i2 -> grid[t][u2][q], q = u1*C + f.
struct InFwdCols {
  const float2* rows;  // (t, 0, q)
  uint32_t step;       // bytes from one row to the next
  __device__ float2 at(int i2, int col) const { return load_at(rows, (uint32_t)i2 * step + (uint32_t)col * 8u); }
};
struct OutFwdCols {
  float2* grid;   // (t, 0, q)
  uint32_t step;  // bytes from one row to the next
  uint64_t used;  // blocks of the column that some sample reads
  __device__ void operator()(int pos, int col, float2 val) const {
    if (used >> (pos / kGridBlock) & 1) store_at(grid, (uint32_t)pos * step + (uint32_t)col * 8u, val);
  }
};
// Adjoint columns: grid[t][u2][q] -> inverse FFT along u2, crop -> rows[t][i2][q].
struct InAdjCols {
  const float2* grid;
  uint32_t step;
  uint64_t used;  // blocks of the column that the spread filled; the others are zero
  __device__ float2 operator()(int pos, int col) const {
    if (!(used >> (pos / kGridBlock) & 1)) return make_float2(0.f, 0.f);
    return load_at(grid, (uint32_t)pos * step + (uint32_t)col * 8u);
  }
};
template <int n>
struct OutAdjCols {
  float2* rows;
  uint32_t step;
  __device__ void operator()(int pos, int col, float2 val) const {
    const int i2 = image_index<n>(pos);
    if (i2 >= 0) at(i2, col, val);
  }
  __device__ void at(int i2, int col, float2 val) const {
    store_at(rows, (uint32_t)i2 * step + (uint32_t)col * 8u, val);
  }
};
// Adjoint rows: rows[t][i2][u1][f] -> inverse FFT along u1, crop,
// * scale c(i1) c(i2) -> out[t][i2][i1][f0 + f].
struct InAdjRows {
  const float2* rows;  // position (row, 0, fbase)
  uint32_t step;
  int live;            // valid bins from fbase on
  __device__ float2 operator()(int pos, int col) const {
    if (col >= live) return make_float2(0.f, 0.f);
    return load_at(rows, (uint32_t)pos * step + (uint32_t)col * 8u);
  }
};
template <int n>
struct OutAdjRows {
  float2* out;  // voxel (t, i2, 0, f0 + fbase)
  const float* dp;
  uint32_t step;
  int live;
  float c2;
  __device__ void operator()(int pos, int col, float2 val) const {
    const int i1 = image_index<n>(pos);
    if (i1 >= 0) at(i1, col, val);
  }
  __device__ void at(int i1, int col, float2 val) const {
    if (col < live) store_at(out, (uint32_t)i1 * step + (uint32_t)col * 8u, cscale(val, dp[i1] * c2));
  }
};

template <int NFFT, int KIND>
constexpr int kValsOf = KIND == kFwdCols || KIND == kAdjCols ? kValsCols<NFFT> : kValsPlain<NFFT>;

// Lines a CTA of these kernels.  The long rows take 8, so that two or three
// CTAs fit an SM and one's loads overlap another's butterflies (16 lines, one
// CTA -> 8 lines: 1024 points 36 -> 32 us forward and 36 -> 30 us adjoint, 768
// points 64 -> 53 us forward at three CTAs, 58 at two; the 768-point adjoint
// pass, which writes half as much as it reads, is better off with 16: 62
// against 66 us).
template <int NFFT, int KIND>
constexpr int kColsOf = (NFFT > 512 && KIND == kFwdRows) || (NFFT == 1024 && KIND == kAdjRows) ? 8 : kFftCols;
template <int NFFT, int KIND>
constexpr int kMinCtasOf = kColsOf<NFFT, KIND> == kFftCols ? 0 : NFFT == 768 ? 3 : 2;
template <int NFFT, int KIND>
constexpr int kThreadsOf = NFFT / kValsOf<NFFT, KIND> * kColsOf<NFFT, KIND>;
template <int NFFT, int KIND>
constexpr size_t kSmemOf = ((size_t)NFFT * kColsOf<NFFT, KIND> + Shape<NFFT, kValsOf<NFFT, KIND>>::TW) * sizeof(float2);

template <int NFFT, int KIND>
__global__ void __launch_bounds__(kThreadsOf<NFFT, KIND>, kMinCtasOf<NFFT, KIND>) fft_kernel(FftArgs a) {
  constexpr int EV = kValsOf<NFFT, KIND>, COLS = kColsOf<NFFT, KIND>;
  constexpr int N = NFFT / 2;
  extern __shared__ float2 smem[];
  float2* X = smem;
  float2* tw = smem + NFFT * COLS;
  build_twiddles<NFFT, EV>(tw, a.twiddle);
  grid_dep_wait();
  grid_dep_release();
  __syncthreads();
  const int col = threadIdx.x % COLS;
  const int tl = line_thread<NFFT, EV, COLS>(threadIdx.x);
  if constexpr (KIND == kFwdRows || KIND == kAdjRows) {
    const size_t row = blockIdx.y;  // t*N + i2
    const int i2 = (int)(row % N);
    const int fbase = blockIdx.x * COLS;
    const size_t wpos = row * NFFT * a.C + fbase, vox = row * N * a.Nf + a.f0 + fbase;
    const uint32_t wstep = (uint32_t)a.C * 8u, vstep = (uint32_t)a.Nf * 8u;
    if constexpr (KIND == kFwdRows) {
      InFwdRows in{a.src + vox, a.deapod, vstep, a.Cv - fbase, a.deapod[i2]};
      OutFwdRows out{a.dst + wpos, wstep, a.C - fbase};
      fft_pass<NFFT, EV, -1, 0, 1, true, false, CtaSync, InFwdRows, OutFwdRows, NoHook, COLS>(X, tw, col, tl, in, out);
    } else {
      InAdjRows in{a.src + wpos, wstep, a.Cv - fbase};
      OutAdjRows<NFFT> out{a.dst + vox, a.deapod, vstep, a.Cv - fbase, a.deapod[i2] * a.scale};
      fft_pass<NFFT, EV, +1, 0, 1, false, true, CtaSync, InAdjRows, OutAdjRows<NFFT>, NoHook, COLS>(X, tw, col, tl, in, out);
    }
  } else {
    const size_t nq = (size_t)NFFT * a.C, q = (size_t)blockIdx.x * kFftCols, t = blockIdx.y;
    const uint32_t step = (uint32_t)(nq * sizeof(float2));
    const uint64_t used = used_blocks(a.used, a.ushift, NFFT, t, blockIdx.x);
    if constexpr (KIND == kFwdCols) {
      InFwdCols in{a.src + t * N * nq + q, step};
      OutFwdCols out{a.dst + t * NFFT * nq + q, step, used};
      fft_pass<NFFT, EV, -1, 0, 1, true, false>(X, tw, col, tl, in, out);
    } else {
      InAdjCols in{a.src + t * NFFT * nq + q, step, used};
      OutAdjCols<NFFT> out{a.dst + t * N * nq + q, step};
      fft_pass<NFFT, EV, +1, 0, 1, false, true>(X, tw, col, tl, in, out);
    }
  }
}

// --- Fused row kernel: inverse row FFT -> TV + Adam -> next forward row FFT --
//
// With the whole bin range in one grid pass, the last adjoint pass (inverse
// FFT along u1, crop, deapodise, scale), the optimiser update and the first
// forward pass of the next iteration (deapodise, pad, FFT along x1) all work
// on the same (t, i2) image row and 16 bins.  One CTA does the three in
// turn: the gradient never goes to global memory, and the row workspace is
// rewritten in place (each CTA reads its slice completely before writing it).
// The arithmetic is that of the separate kernels, so the iterates are the
// same bit for bit.  With kRowGrad it stops at the gradient of the loss, for
// callers with an optimiser of their own (fused_rows_grad_pays: where).
struct FusedArgs {
  float2* rows;        // [T][N][n][C] in: adjoint row intermediate, out: next forward row intermediate
  const float* deapod;
  const float2* twiddle;
  const float2* Vin;
  float2* Vout;
  float2* m;
  float2* v;
  double* partials;
  unsigned int* counter;
  const double* data_loss;
  double* loss_out;
  int N, Nf, C, T;
  float scale;         // adjoint scale (1/N)
  AdamArgs ad;
  // warp-specialised kernel only
  int* err;            // device status word (bounded wait expired)
  int units;           // (t, i2, 16-bin) row units, unit = (t N + i2) nfb + bin group
  int nfb;             // 16-bin groups per image row
  int bh, nbox;        // tensor-copy box height and boxes per unit
};

// Kernel parameter of the fused row kernel over a batch of problems.
struct MultiFused {
  FusedArgs a[kMaxBatch];
  int fwd_tail[kMaxBatch];
  int nreq;
  int unit_begin[kMaxBatch + 1];   // unit (block) ranges of the problems
};

// Adjoint output into the CTA's gradient buffer gb[i1][col].
template <int n>
struct OutGrad {
  float2* gb;
  const float* dp;
  float c2;
  __device__ void operator()(int pos, int col, float2 val) const {
    const int i1 = image_index<n>(pos);
    if (i1 >= 0) gb[i1 * kFftCols + col] = cscale(val, dp[i1] * c2);
  }
  __device__ void at(int i1, int col, float2 val) const { gb[i1 * kFftCols + col] = cscale(val, dp[i1] * c2); }
};
// Forward input from the CTA's new-volume buffer vb[i1][col].
struct InNewRow {
  const float2* vb;
  const float* dp;
  float c2;
  __device__ float2 at(int i1, int col) const { return cscale_rn(vb[i1 * kFftCols + col], dp[i1] * c2); }
};

// TV + Adam on the (t, i2) image row, bins fbase .. fbase + 15.  The
// nthreads threads split the row into 16 columns (one bin each) of
// nthreads / 16 runs of consecutive i1; thread tid walks its run, so the
// x1 neighbours are the previous and the next voxel of the walk and only the
// next one is loaded per step.  The adjoint gradient comes from gb[i1][col],
// the new value goes to Vout and back into gb (zero for bins >= Nf, the
// padding of the next forward row transform).  Adds this thread's TV shares
// to `local` in walk order and returns it.  The walk goes U voxels at a time:
// all their loads are issued before the first is used (left to the compiler,
// the stores of one voxel held back the loads of the next, and a voxel cost
// 3000 clocks of load latency).  Every load is unconditional (missing
// neighbours and bins >= Nf read a valid voxel whose value is then not used).
// TT: the volume has time neighbours (T > 1 and tv_t != 0).  Without ADAM the
// gradient itself goes to Vout, gb stays as it is.
template <bool TT, bool ADAM, int U>
__device__ __forceinline__ float update_row(const FusedArgs& a, float2* gb, int i2, int t, int fbase, int tid,
                                            int nthreads, float local) {
  const float eps2 = a.ad.tv_eps * a.ad.tv_eps;
  // The volumes and moments never alias: loads of later voxels may be issued
  // ahead of the stores of earlier ones.
  const float2* __restrict__ Vin = a.Vin;
  float2* __restrict__ Vout = a.Vout;
  float2* __restrict__ mom1 = a.m;
  float2* __restrict__ mom2 = a.v;
  const int col = tid % kFftCols;
  const int runs = nthreads / kFftCols;
  const int len = (a.N + runs - 1) / runs;
  const int lo = (tid / kFftCols) * len;
  const int hi = min(a.N, lo + len);
  if (lo >= hi) return local;
  const size_t sy = (size_t)a.N * a.Nf, st = (size_t)a.N * a.N * a.Nf;
  const bool xy = a.ad.tv_xy != 0.f;
  const bool h2p = xy && i2 + 1 < a.N, h2m = xy && i2 > 0;
  const bool htp = TT && t + 1 < a.T, htm = TT && t > 0;
  const int f = fbase + col;
  const bool fv = f < a.Nf;
  // A voxel is one 32-bit byte offset into each array, from the frame before
  // the unit's (its own when t = 0); the neighbouring rows and frames are
  // fixed distances from it, 0 for a missing one (this voxel is read).
  const size_t first = (size_t)(t > 0 ? t - 1 : 0) * st;
  const float2* rx = Vin + first;
  float2* rm = mom1 + first;
  float2* rv = mom2 + first;
  float2* ro = Vout + first;
  const uint32_t sx = (uint32_t)a.Nf * 8u;
  const uint32_t d2 = (uint32_t)sy * 8u, dt = (uint32_t)st * 8u;
  const uint32_t d2p = h2p ? d2 : 0u, d2m = h2m ? d2 : 0u, dtp = htp ? dt : 0u, dtm = htm ? dt : 0u;
  uint32_t off = (t > 0 ? dt : 0u) + (uint32_t)i2 * d2 + (uint32_t)lo * sx + (uint32_t)(fv ? f : a.Nf - 1) * 8u;
  auto at = [](const float2* b, uint32_t o) {
    return load_at(b, o);  // (Vin is not written by this kernel)
  };
  const float tv_xy = a.ad.tv_xy, tv_t = TT ? a.ad.tv_t : 0.f;
  float2 x = at(rx, off);
  // The TV term of the difference from the voxel before: it is that voxel's
  // own term towards this one, computed once and handed on along the walk.
  float mag;
  float2 g1m = make_float2(0.f, 0.f);
  if (xy && lo > 0) g1m = tv_term(csub_rn(x, at(rx, off - sx)), eps2, &mag);
  for (int i0 = lo; i0 < hi; i0 += U, off += U * sx) {
    // every load of U voxels before the first use of one
    float2 xp[U], x2p[U], x2m[U], xtp[U], xtm[U], mm[U], vv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t o = off + (uint32_t)min(u, hi - 1 - i0) * sx;
      xp[u] = at(rx, min(i0 + u, hi - 1) + 1 < a.N ? o + sx : o);
      x2p[u] = at(rx, o + d2p);
      x2m[u] = at(rx, o - d2m);
      if constexpr (TT) {
        xtp[u] = at(rx, o + dtp);
        xtm[u] = at(rx, o - dtm);
      }
      if constexpr (ADAM) {
        mm[u] = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(rm) + o);
        vv[u] = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(rv) + o);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i1 = i0 + u;
      if (i1 >= hi) break;
      const uint32_t o = off + (uint32_t)u * sx;
      float2* gp = gb + i1 * kFftCols + col;
      const float2 gd = *gp;
      // voxel_tv_nb's terms in its order
      float2 gxy = make_float2(0.f, 0.f), gt = make_float2(0.f, 0.f), g1p = make_float2(0.f, 0.f);
      float sxy = 0.f, stt = 0.f;
      if (xy) {
        if (i1 + 1 < a.N) {
          g1p = tv_term(csub_rn(xp[u], x), eps2, &mag);
          gxy = csub_rn(gxy, g1p);
          sxy = __fadd_rn(sxy, mag);
        }
        if (i1 > 0) gxy = cadd_rn(gxy, g1m);
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
      float2 nx = make_float2(0.f, 0.f);
      if (fv) {
        local = __fadd_rn(local, fmaf(tv_xy, sxy, __fmul_rn(tv_t, stt)));
        const float2 g = total_grad(gd, gxy, gt, a.ad);
        if constexpr (ADAM) {
          nx = adam_voxel(x, g, mm[u], vv[u], a.ad);
          store_at(rm, o, mm[u]);
          store_at(rv, o, vv[u]);
          store_at(ro, o, nx);
        } else {
          store_at(ro, o, g);
        }
      }
      if constexpr (ADAM) *gp = nx;
      g1m = g1p;
      x = xp[u];
    }
  }
  return local;
}

// UT, UP: voxels whose loads are issued together with and without time
// neighbours, as many as the caller's registers hold.
template <bool ADAM, int UT, int UP>
__device__ __forceinline__ float update_row_any(const FusedArgs& a, float2* gb, int i2, int t, int fbase, int tid,
                                                int nthreads, float local) {
  if (a.T > 1 && a.ad.tv_t != 0.f) return update_row<true, ADAM, UT>(a, gb, i2, t, fbase, tid, nthreads, local);
  return update_row<false, ADAM, UP>(a, gb, i2, t, fbase, tid, nthreads, local);
}

// L2 prefetch of the update's Adam moments for image row `row`.  (The rows of
// V are read by their neighbours' updates at about the same time; prefetching
// them too cost more L2 requests than it hid: dynamic 375 against 369 us.)
__device__ __forceinline__ void prefetch_update_rows(const FusedArgs& a, size_t row) {
  const size_t rl = (size_t)a.N * a.Nf;
  const uint32_t rb = (uint32_t)(rl * sizeof(float2));
  prefetch_l2(a.m + row * rl, rb);
  prefetch_l2(a.v + row * rl, rb);
}

// Register cap: 64 a thread (two CTAs of 512 threads per SM); above 512 points
// one CTA of 512 threads fits the shared memory.
template <int NFFT>
constexpr int fused_min_blocks() {
  return NFFT > 512 ? 1 : 65536 / (Shape<NFFT, kValsFused<NFFT>>::THREADS * 64) > 16
             ? 16
             : 65536 / (Shape<NFFT, kValsFused<NFFT>>::THREADS * 64);
}

// The fused row kernel's work on one (image row, 16-bin group) unit: bin
// group bx of image row `row` (t N + i2); vb, nblk: the unit's index and the
// unit count of the loss reduction.
// What the fused row kernel does after the inverse FFT of its row.
enum RowMode { kRowUpdate = 0, kRowUpdateFwd = 1, kRowGrad = 2 };  // Adam; Adam and the next forward FFT; gradient only

// Transform lengths with a kRowGrad kernel.
constexpr bool row_grad_size(int n) { return n >= 48 && n <= 768; }

template <int NFFT, int MODE>
__device__ __forceinline__ void fused_rows_body(const FusedArgs& a, int bx, size_t row, unsigned vb, unsigned nblk) {
  constexpr int EV = kValsFused<NFFT>;
  extern __shared__ float2 smem[];
  float2* X = smem;
  float2* tw = smem + NFFT * kFftCols;
  float2* gb = tw + Shape<NFFT, EV>::TW;  // [N][kFftCols]
  const int i2 = (int)(row % a.N);
  const int t = (int)(row / a.N);
  build_twiddles<NFFT, EV>(tw, a.twiddle);
  grid_dep_wait();
  grid_dep_release();
  // the update's operands stream into L2 while the inverse FFT runs
  constexpr bool ADAM = MODE != kRowGrad;
  if (ADAM && threadIdx.x == 0) prefetch_update_rows(a, row);
  __syncthreads();
  const int col = threadIdx.x % kFftCols;
  const int tl = line_thread<NFFT, EV>(threadIdx.x);
  const int fbase = bx * kFftCols;
  float2* wpos = a.rows + row * NFFT * a.C + fbase;
  const uint32_t wstep = (uint32_t)a.C * 8u;
  {
    InAdjRows in{wpos, wstep, a.Nf - fbase};
    OutGrad<NFFT> out{gb, a.deapod, a.deapod[i2] * a.scale};
    fft_pass<NFFT, EV, +1, 0, 1, false, true>(X, tw, col, tl, in, out);
  }
  __syncthreads();
  const float local = update_row_any<ADAM, ADAM ? 2 : 3, ADAM ? 2 : 4>(a, gb, i2, t, fbase, threadIdx.x, blockDim.x, 0.f);
  if constexpr (MODE == kRowUpdateFwd) {
    __syncthreads();
    InNewRow in{gb, a.deapod, a.deapod[i2]};
    OutFwdRows out{wpos, wstep, a.C - fbase};
    fft_pass<NFFT, EV, -1, 0, 1, true, false>(X, tw, col, tl, in, out);
  }
  finish_loss_v(local, a.partials, a.counter, a.data_loss, a.loss_out, vb, nblk);
}

template <int NFFT, int MODE>
__global__ void __launch_bounds__(Shape<NFFT, kValsFused<NFFT>>::THREADS, fused_min_blocks<NFFT>())
    fused_rows_kernel(FusedArgs a) {
  fused_rows_body<NFFT, MODE>(a, blockIdx.x, blockIdx.y, blockIdx.y * gridDim.x + blockIdx.x,
                                  gridDim.x * gridDim.y);
}

// One launch of the fused row kernel for several problems of the same
// transform length (a batch of requests): block b serves problem r with
// unit_begin[r] <= b < unit_begin[r + 1], unit u = b - unit_begin[r] =
// (image row) nfb + bin group, the same unit and loss-partial order as the
// problem's own launch, so every result is the same bit for bit.
template <int NFFT>
__global__ void __launch_bounds__(Shape<NFFT, kValsFused<NFFT>>::THREADS, fused_min_blocks<NFFT>())
    fused_rows_multi_kernel(const __grid_constant__ MultiFused m) {
  int r = 0;
  while (r + 1 < m.nreq && (int)blockIdx.x >= m.unit_begin[r + 1]) ++r;
  const unsigned u = blockIdx.x - (unsigned)m.unit_begin[r];
  const unsigned nu = (unsigned)(m.unit_begin[r + 1] - m.unit_begin[r]);
  const FusedArgs& a = m.a[r];
  const int bx = (int)(u % (unsigned)a.nfb);
  const size_t row = u / (unsigned)a.nfb;
  if (m.fwd_tail[r])
    fused_rows_body<NFFT, kRowUpdateFwd>(a, bx, row, u, nu);
  else
    fused_rows_body<NFFT, kRowUpdate>(a, bx, row, u, nu);
}

template <int NFFT>
size_t fused_smem(int N) {
  return Shape<NFFT, kValsFused<NFFT>>::SMEM + (size_t)N * kFftCols * sizeof(float2);
}

template <int NFFT>
cudaError_t launch_fused_multi(const MultiFused& m, cudaStream_t s) {
  const size_t smem = fused_smem<NFFT>(m.a[0].N);
  for (int r = 1; r < m.nreq; ++r)
    if (m.a[r].N != m.a[0].N) return cudaErrorInvalidValue;
  return launch_dep(fused_rows_multi_kernel<NFFT>, dim3((unsigned)m.unit_begin[m.nreq]),
                    dim3(Shape<NFFT, kValsFused<NFFT>>::THREADS), smem, s, m);
}

template <int NFFT>
cudaError_t launch_fused(const FusedArgs& a, int mode, dim3 grid, cudaStream_t s) {
  const size_t smem = fused_smem<NFFT>(a.N);
  const dim3 block(Shape<NFFT, kValsFused<NFFT>>::THREADS);
  if (mode == kRowGrad) {
    if constexpr (row_grad_size(NFFT)) return launch_dep(fused_rows_kernel<NFFT, kRowGrad>, grid, block, smem, s, a);
    return cudaErrorInvalidValue;
  }
  if (mode == kRowUpdateFwd) return launch_dep(fused_rows_kernel<NFFT, kRowUpdateFwd>, grid, block, smem, s, a);
  return launch_dep(fused_rows_kernel<NFFT, kRowUpdate>, grid, block, smem, s, a);
}

// --- Warp-specialised fused row kernel ---------------------------------------
//
// Persistent CTAs (one per SM) walk the row units u = blockIdx.x + i
// gridDim.x.  The first FT threads (the transform group, one FFT tile's
// worth) run, for i = 0, 1, ...: the inverse row FFT of unit i into
// gradient buffer i % 2, then the forward row FFT of unit i - 1 from buffer
// (i - 1) % 2; the other kUpdThreads threads (the update group) meanwhile
// apply TV + Adam to unit i - 1 .. i in place in its buffer.  The update's
// HBM stream of V, m and v thus overlaps the transforms' shared-memory work
// instead of following it.  The adjoint input of unit i + 1 is staged by a
// tensor copy as soon as the first pass of unit i has read the stage.
// Hand-offs: ready[b] (every transform thread arrives once the inverse FFT
// has written buffer b) and done[b] (every update thread arrives once it
// has rewritten buffer b); each group synchronises internally on its own
// named barrier.  A group gives up on an expired bounded wait (the status
// word is set); the other group's next wait then expires too.  The
// arithmetic is that of fused_rows_kernel, so the iterates agree bit for
// bit; the TV partial sums are per CTA.
constexpr int kUpdThreads = 512;

// Input staged in shared memory as [rows][kFftCols].
struct InTile {
  const float2* t;  // [rows][kFftCols]
  __device__ float2 at(int i, int col) const { return t[i * kFftCols + col]; }
  __device__ float2 operator()(int pos, int col) const { return t[pos * kFftCols + col]; }
};

template <int NFFT>
constexpr bool fused_ws_fits() {
  return NFFT <= 512 && Shape<NFFT, kValsFused<NFFT>>::THREADS % 32 == 0 && Shape<NFFT, kValsFused<NFFT>>::THREADS <= 512;
}

template <int NFFT>
constexpr size_t fused_ws_smem() {
  // stage + transform workspace [NFFT][16], two gradient buffers [N][16], twiddles, 5 mbarriers
  return (size_t)2 * NFFT * kFftCols * sizeof(float2) + (size_t)2 * (NFFT / 2) * kFftCols * sizeof(float2) +
         (size_t)Shape<NFFT, kValsFused<NFFT>>::TW * sizeof(float2) + 5 * sizeof(uint64_t);
}

template <int NFFT, bool FWD_TAIL>
__global__ void __launch_bounds__(Shape<NFFT, kValsFused<NFFT>>::THREADS + kUpdThreads, 1)
    fused_rows_ws_kernel(const __grid_constant__ CUtensorMap tin, FusedArgs a) {
  constexpr int EV = kValsFused<NFFT>;
  constexpr int FT = Shape<NFFT, EV>::THREADS;
  using FSync = GroupSync<1, FT>;
  using USync = GroupSync<2, kUpdThreads>;
  extern __shared__ __align__(128) float2 smem[];
  float2* S = smem;                          // [NFFT][16] staged adjoint input
  float2* X = S + NFFT * kFftCols;           // [NFFT][16] transform workspace
  float2* gbuf = X + NFFT * kFftCols;        // [2][N][16]
  float2* tw = gbuf + 2 * (NFFT / 2) * kFftCols;
  uint64_t* full = reinterpret_cast<uint64_t*>(tw + Shape<NFFT, EV>::TW);
  uint64_t* ready = full + 1;                // [2]
  uint64_t* done = full + 3;                 // [2]
  __shared__ volatile int s_abort_f, s_abort_u;
  const int nu = (int)blockIdx.x < a.units ? (a.units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const int gsz = a.N * kFftCols;
  const uint32_t tile_bytes = (uint32_t)(NFFT * kFftCols * sizeof(float2));
  auto issue = [&](int i) {
    const int u = (int)blockIdx.x + i * (int)gridDim.x;
    const int row = u / a.nfb, fb = u - (u / a.nfb) * a.nfb;
    mbar_expect_tx(full, tile_bytes);
    for (int b = 0; b < a.nbox; ++b)
      tma_load_3d(S + (size_t)b * a.bh * kFftCols, &tin, fb * 2 * kFftCols, b * a.bh, row, full);
  };
  if (threadIdx.x == 0) {
    mbar_init(full, 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&ready[b], FT);
      mbar_init(&done[b], kUpdThreads);
    }
    fence_mbar_init();
    s_abort_f = 0;
    s_abort_u = 0;
  }
  build_twiddles<NFFT, EV>(tw, a.twiddle);
  grid_dep_wait();
  grid_dep_release();
  int issued = 0, consumed = 0;  // tensor copies, meaningful on thread 0
  if (threadIdx.x == 0 && nu > 0) {
    issue(0);
    issued = 1;
  }
  __syncthreads();
  float local = 0.f;
  // The update's loads in flight are what its registers hold, so it takes
  // part of the transform group's (whole warpgroups; the shares of both
  // groups add up to the launch's 64 a thread): 80 a thread hold three
  // voxels' loads with time neighbours where 64 spilled at two.  Together
  // with those loads issued at once: dynamic 445 -> 370 us.
  // A walk that three voxels at a time do not shorten takes two, and a walk of
  // one voxel (N <= 32) one: the rest of a step would load its last voxel again.
  constexpr int LEN = (NFFT / 2 + kUpdThreads / kFftCols - 1) / (kUpdThreads / kFftCols);
  constexpr int UP = LEN < 2 ? LEN : 2, UT = (LEN + 2) / 3 < (LEN + 1) / 2 ? 3 : UP;
  constexpr bool SPLIT = FT == kUpdThreads;
  constexpr int FREG = EV == 12 ? 48 : 56;  // fused_ws_runs checks the launch's registers
  if (threadIdx.x < FT) {
    if constexpr (SPLIT) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(FREG));
    const int col = threadIdx.x % kFftCols;
    const int tl = line_thread<NFFT, EV>(threadIdx.x);
    for (int i = 0; i <= nu; ++i) {
      if (i < nu) {
        if (!mbar_wait_bounded(full, (uint32_t)(i & 1)))
          s_abort_f = 1;
        else
          ++consumed;
        FSync::sync();  // the previous forward FFT is done with X; uniform abort flag
        if (s_abort_f) break;
        const int u = (int)blockIdx.x + i * (int)gridDim.x;
        const size_t row = (size_t)(u / a.nfb);
        const int i2 = (int)(row % a.N);
        auto hook = [&]() {
          if (threadIdx.x == 0 && i + 1 < nu) {
            fence_proxy_async_smem();
            issue(i + 1);
            ++issued;
          }
        };
        InTile in{S};
        OutGrad<NFFT> out{gbuf + (size_t)(i & 1) * gsz, a.deapod, a.deapod[i2] * a.scale};
        fft_pass<NFFT, EV, +1, 0, 1, false, true, FSync>(X, tw, col, tl, in, out, hook);
        mbar_arrive(&ready[i & 1]);
      }
      if (i >= 1) {
        const int j = i - 1;
        if (!mbar_wait_bounded(&done[j & 1], (uint32_t)((j >> 1) & 1))) s_abort_f = 1;
        FSync::sync();  // the inverse FFT's last pass is done with X; uniform abort flag
        if (s_abort_f) break;
        if constexpr (FWD_TAIL) {
          const int u = (int)blockIdx.x + j * (int)gridDim.x;
          const size_t row = (size_t)(u / a.nfb);
          const int fbase = (u - (u / a.nfb) * a.nfb) * kFftCols;
          const int i2 = (int)(row % a.N);
          InNewRow in{gbuf + (size_t)(j & 1) * gsz, a.deapod, a.deapod[i2]};
          OutFwdRows out{a.rows + row * NFFT * a.C + fbase, (uint32_t)a.C * 8u, a.C - fbase};
          fft_pass<NFFT, EV, -1, 0, 1, true, false, FSync>(X, tw, col, tl, in, out);
        }
      }
    }
  } else {
    if constexpr (SPLIT) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(128 - FREG));
    const int ut = threadIdx.x - FT;
    if (ut == 0 && nu > 0) {
      prefetch_update_rows(a, (size_t)(blockIdx.x / a.nfb));
    }
    for (int i = 0; i < nu; ++i) {
      const int u = (int)blockIdx.x + i * (int)gridDim.x;
      const size_t row = (size_t)(u / a.nfb);
      const int fbase = (u - (u / a.nfb) * a.nfb) * kFftCols;
      const int i2 = (int)(row % a.N), t = (int)(row / a.N);
      if (ut == 0 && i + 1 < nu) {
        const size_t nrow = (size_t)((u + (int)gridDim.x) / a.nfb);
        if (nrow != row) prefetch_update_rows(a, nrow);
      }
      if (!mbar_wait_bounded(&ready[i & 1], (uint32_t)((i >> 1) & 1))) s_abort_u = 1;
      USync::sync();
      if (s_abort_u) break;
      local = update_row_any<true, UT, UP>(a, gbuf + (size_t)(i & 1) * gsz, i2, t, fbase, ut, kUpdThreads, local);
      mbar_arrive(&done[i & 1]);
    }
  }
  __syncthreads();
  if ((s_abort_f || s_abort_u) && threadIdx.x == 0) {
    atomicExch(a.err, 1);
    // let copies issued and never awaited land (bounded)
    for (int k = consumed; k < issued; ++k) mbar_wait_bounded(full, (uint32_t)(k & 1));
  }
  finish_loss(local, a.partials, a.counter, a.data_loss, a.loss_out);
}

template <int NFFT>
cudaError_t launch_fused_ws(const CUtensorMap& tm, const FusedArgs& a, bool fwd_tail, int ctas, cudaStream_t s) {
  if constexpr (fused_ws_fits<NFFT>()) {
    const dim3 grid((unsigned)ctas), block(Shape<NFFT, kValsFused<NFFT>>::THREADS + kUpdThreads);
    if (fwd_tail) return launch_dep(fused_rows_ws_kernel<NFFT, true>, grid, block, fused_ws_smem<NFFT>(), s, tm, a);
    return launch_dep(fused_rows_ws_kernel<NFFT, false>, grid, block, fused_ws_smem<NFFT>(), s, tm, a);
  } else {
    return cudaErrorInvalidValue;
  }
}

// --- Column passes staged by TMA ------------------------------------------
//
// Persistent CTAs walk the column tiles (16 adjacent (u1, bin) lines of one
// frame); the next tile for a buffer is loaded by a tensor copy as soon as
// the first pass of the tile in it has read it, so the input of the next
// tiles streams in while this one is transformed.
// Forward: the staged input is the N image rows of the row intermediate
// (padding is never stored); adjoint: the 2N grid rows.  Of the grid only the
// blocks that samples reach (Plan::grid_used) are written (forward) or copied
// in (adjoint: a box without such a block is requested outside the tensor, so
// that the copy fills it with zeros and reads nothing).
struct ColArgs {
  float2* dst;
  const float2* twiddle;
  int* err;
  size_t nq;
  int qtiles, ntiles, bh, nbox;
  const uint64_t* used;  // grid blocks in use [frame][u1 / 2], or null
  int ushift;            // log2 of the 16-line tiles in two grid columns
  uint64_t box_mask;     // adjoint: the grid blocks in one box, at bit 0
};

// Kernel parameter of a column pass over a batch of problems.
struct MultiCols {
  CUtensorMap tm[kMaxBatch];       // each problem's input tensor map
  ColArgs a[kMaxBatch];
  int nreq;
  int cta_begin[kMaxBatch + 1];    // CTA ranges of the problems
};

template <int NFFT, int KIND>
constexpr int col_rows() {
  return KIND == kFwdCols ? NFFT / 2 : NFFT;
}
// Tile buffers and CTAs per SM: the forward pass stages the N image rows in
// one buffer (the next tile is requested once the first pass has read the
// current one) with two CTAs per SM up to 2N = 512 and one above (two would
// not fit the shared memory, and their bound on the registers made 1024
// threads spill); the adjoint stages all 2N rows, in one buffer with two CTAs
// per SM where two such CTAs fit an SM's shared memory (2N <= 384), double-
// buffered with one CTA per SM at 512, in one buffer at 768 (at 1024 a tile
// beside the exchange buffer does not fit: unstaged).
template <int NFFT, int KIND>
constexpr int col_bufs() {
  return KIND == kAdjCols && NFFT == 512 ? 2 : 1;
}
template <int NFFT, int KIND>
constexpr int col_ctas_per_sm() {
  return NFFT <= (KIND == kFwdCols ? 512 : 384) ? 2 : 1;
}
template <int NFFT, int KIND>
constexpr size_t col_smem() {
  return (size_t)col_bufs<NFFT, KIND>() * col_rows<NFFT, KIND>() * kFftCols * sizeof(float2) +
         Shape<NFFT, kValsCols<NFFT>>::SMEM + 2 * sizeof(uint64_t);
}

// Shared memory of a launch of `ctas` persistent CTAs over ntiles tiles.  The
// launch may find SMs still held by the kernel before it; a CTA of a short
// transform leaves room for many, so the free SMs would then take more than
// their share of the CTAs and the pass would last as long as the fullest SM.
// From two tiles a CTA on, a launch therefore asks for so much that no SM holds
// more than its share (32 frames of 32^2 x 32 bins: forward 37.2 -> 30.6 us,
// gradient 137 -> 123, an iteration 12.5 -> 10.7; 32 frames of 64^2 x 64 bins:
// an iteration 79 -> 72 us).  Below that the CTAs are over before it matters and
// early ones beside the spread's are worth more (64^2 x 64 bins: 7.1 us an
// iteration, 7.4 with it).
template <int NFFT, int KIND>
size_t col_launch_smem(int ctas, int ntiles) {
  const size_t share = (size_t)228 * 1024 / (col_ctas_per_sm<NFFT, KIND>() + 1);
  return ntiles > 2 * ctas ? std::max(col_smem<NFFT, KIND>(), share) : col_smem<NFFT, KIND>();
}

// The column pass of one problem run by vg persistent CTAs, this being the
// vb-th: tile vb, vb + vg, ... ; tin is the problem's input tensor map (in
// the kernel's parameter space).
template <int NFFT, int KIND>
__device__ __forceinline__ void cols_body(const CUtensorMap* tin, const ColArgs& a, int vb, int vg) {
  constexpr int EV = kValsCols<NFFT>;
  constexpr int H = col_rows<NFFT, KIND>();
  constexpr int NB = col_bufs<NFFT, KIND>();
  extern __shared__ __align__(128) float2 smem[];
  float2* tiles = smem;                      // [NB][H][kFftCols]
  float2* X = tiles + NB * H * kFftCols;     // [NFFT][kFftCols]
  float2* tw = X + NFFT * kFftCols;
  uint64_t* full = reinterpret_cast<uint64_t*>(tw + Shape<NFFT, EV>::TW);
  __shared__ volatile int s_abort;
  const uint32_t tile_bytes = (uint32_t)(H * kFftCols * sizeof(float2));
  // A tile of this CTA: frame, 16-line tile of it, its column's blocks in use.
  struct Tile {
    int t, qt;
    uint64_t used;
  };
  // The CTA's tiles are vg apart: (frame, tile) steps by (step_t, step_q) with
  // one carry instead of a division by every thread for every tile.
  const int step_t = vg / a.qtiles, step_q = vg - step_t * a.qtiles;
  auto advance = [&](int& t, int& qt) {
    t += step_t;
    qt += step_q;
    if (qt >= a.qtiles) {
      qt -= a.qtiles;
      ++t;
    }
  };
  // Whole CTA: request the copy of a tile into buffer b, the boxes dealt out
  // over the warps (a warp issues its boxes one after the other, and the other
  // warps would wait for it at the next barrier).  A box that lands before
  // thread 0 has stated the bytes is made up for by it: the phase cannot end
  // before that arrival.
  constexpr int WARPS = Shape<NFFT, EV>::THREADS >= 32 ? Shape<NFFT, EV>::THREADS / 32 : 1;
  auto issue = [&](const Tile& x, int b) {
    if (threadIdx.x == 0) mbar_expect_tx(&full[b], tile_bytes);
    for (int i = (threadIdx.x % 32) * WARPS + threadIdx.x / 32; i < a.nbox; i += 32 * WARPS) {
      const bool want = KIND == kFwdCols || (x.used >> (i * a.bh / kGridBlock) & a.box_mask) != 0;
      tma_load_3d(tiles + ((size_t)b * H + (size_t)i * a.bh) * kFftCols, tin, x.qt * 2 * kFftCols,
                  want ? i * a.bh : NFFT, x.t, &full[b]);
    }
  };
  if (threadIdx.x == 0) {
    for (int b = 0; b < NB; ++b) mbar_init(&full[b], 1);
    fence_mbar_init();
    s_abort = 0;
  }
  build_twiddles<NFFT, EV>(tw, a.twiddle);
  int nt = vb / a.qtiles, nq = vb - nt * a.qtiles;  // the next tile to request
  Tile tile_of[NB];                                 // of the tiles in the buffers, the current one's first
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    tile_of[b] = Tile{nt, nq, vb + b * vg < a.ntiles ? used_blocks(a.used, a.ushift, NFFT, nt, nq) : 0};
    advance(nt, nq);
  }
  grid_dep_wait();
  grid_dep_release();
  __syncthreads();  // the barriers are initialised before any warp issues on them
#pragma unroll
  for (int b = 0; b < NB; ++b)
    if (vb + b * vg < a.ntiles) issue(tile_of[b], b);
  const int col = threadIdx.x % kFftCols;
  const int tl = line_thread<NFFT, EV>(threadIdx.x);
  const uint32_t step = (uint32_t)(a.nq * sizeof(float2));
  int k = 0;
  for (int tile = vb; tile < a.ntiles; tile += vg, ++k) {
    const int b = k % NB;
    if (!mbar_wait_bounded(&full[b], (uint32_t)((k / NB) & 1))) s_abort = 1;
    __syncthreads();  // the previous tile's last pass is done with X; all threads see s_abort
    if (s_abort) break;
    const size_t t = (size_t)tile_of[0].t, q = (size_t)tile_of[0].qt * kFftCols;
    const bool more = tile + NB * vg < a.ntiles;
    const Tile next{nt, nq, more ? used_blocks(a.used, a.ushift, NFFT, nt, nq) : 0};
    auto hook = [&]() {
      if (more) {
        fence_proxy_async_smem();
        issue(next, b);
      }
    };
    InTile in{tiles + (size_t)b * H * kFftCols};
    if constexpr (KIND == kFwdCols) {
      OutFwdCols out{a.dst + t * NFFT * a.nq + q, step, tile_of[0].used};
      fft_pass<NFFT, EV, -1, 0, 1, true, false>(X, tw, col, tl, in, out, hook);
    } else {
      OutAdjCols<NFFT> out{a.dst + t * (NFFT / 2) * a.nq + q, step};
      fft_pass<NFFT, EV, +1, 0, 1, false, true>(X, tw, col, tl, in, out, hook);
    }
#pragma unroll
    for (int i = 0; i + 1 < NB; ++i) tile_of[i] = tile_of[i + 1];
    tile_of[NB - 1] = next;
    advance(nt, nq);
  }
  if (s_abort && threadIdx.x == 0) {
    atomicExch(a.err, 1);
    // let copies this CTA issued and nobody consumed land (bounded)
    for (int kk = k; kk < k + NB; ++kk)
      if (vb + kk * vg < a.ntiles) mbar_wait_bounded(&full[kk % NB], (uint32_t)((kk / NB) & 1));
  }
}

template <int NFFT, int KIND>
__global__ void __launch_bounds__(Shape<NFFT, kValsCols<NFFT>>::THREADS, col_ctas_per_sm<NFFT, KIND>())
    fft_cols_tma_kernel(const __grid_constant__ CUtensorMap tin, ColArgs a) {
  cols_body<NFFT, KIND>(&tin, a, blockIdx.x, gridDim.x);
}

// One launch of a column pass for several problems of the same transform
// length: CTA b serves problem r with cta_begin[r] <= b < cta_begin[r + 1],
// as CTA b - cta_begin[r] of cta_begin[r + 1] - cta_begin[r].  Every tile is
// transformed exactly as by the problem's own launch.
template <int NFFT, int KIND>
__global__ void __launch_bounds__(Shape<NFFT, kValsCols<NFFT>>::THREADS, col_ctas_per_sm<NFFT, KIND>())
    fft_cols_multi_kernel(const __grid_constant__ MultiCols m) {
  int r = 0;
  while (r + 1 < m.nreq && (int)blockIdx.x >= m.cta_begin[r + 1]) ++r;
  cols_body<NFFT, KIND>(&m.tm[r], m.a[r], (int)blockIdx.x - m.cta_begin[r], m.cta_begin[r + 1] - m.cta_begin[r]);
}

// The same for the plain passes, whose CTAs are few where a problem is small: up
// to four an SM, a launch asks for so much shared memory that no SM takes more
// than its share (forward passes one after the other: 64^2 x 16 bins 14.2 ->
// 11.4 us, 8 frames of 32^2 x 32 bins 14.8 -> 12.4; adjoint of 96^2 x 64 bins
// 38.1 -> 31.2).  Fewer CTAs than a quarter of the SMs spread by themselves, and
// start later if they have to wait for an empty SM (32^2 x 8 bins 7.9 us, 7.5
// without; from 48 CTAs on, 48^2 x 8 bins 8.4 and 10.0).
constexpr size_t kEvenShare = (size_t)228 * 1024 / 2;  // the most that is asked for: one CTA an SM

template <int NFFT>
cudaError_t launch(int kind, const FftArgs& a, dim3 grid, int sms, cudaStream_t s) {
  auto go = [&](auto kern, int lines, int threads, size_t smem) {
    const dim3 g((grid.x + lines - 1) / lines, grid.y);
    const size_t ctas = (size_t)g.x * g.y, share = (ctas + sms - 1) / sms;
    if (4 * ctas > (size_t)sms && share <= 4) smem = std::max(smem, (size_t)228 * 1024 / (share + 1));
    return launch_dep(kern, g, dim3(threads), smem, s, a);
  };
#define PROP_GO(K) go(fft_kernel<NFFT, K>, kColsOf<NFFT, K>, kThreadsOf<NFFT, K>, kSmemOf<NFFT, K>)
  switch (kind) {
    case kFwdRows: return PROP_GO(kFwdRows);
    case kFwdCols: return PROP_GO(kFwdCols);
    case kAdjCols: return PROP_GO(kAdjCols);
    default: return PROP_GO(kAdjRows);
  }
#undef PROP_GO
}

template <int NFFT>
cudaError_t configure_n() {
  cudaError_t e;
  auto smem = [](auto kern, size_t bytes) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  if ((e = smem(fft_kernel<NFFT, kFwdRows>, std::max(kEvenShare, kSmemOf<NFFT, kFwdRows>)))) return e;
  if ((e = smem(fft_kernel<NFFT, kFwdCols>, std::max(kEvenShare, kSmemOf<NFFT, kFwdCols>)))) return e;
  if ((e = smem(fft_kernel<NFFT, kAdjCols>, std::max(kEvenShare, kSmemOf<NFFT, kAdjCols>)))) return e;
  if ((e = smem(fft_kernel<NFFT, kAdjRows>, std::max(kEvenShare, kSmemOf<NFFT, kAdjRows>)))) return e;
  int optin = 0, dev = 0;
  if ((e = cudaGetDevice(&dev))) return e;
  if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev))) return e;
  const size_t room = (size_t)optin - 1024;
  if (col_smem<NFFT, kFwdCols>() <= room) {
    const size_t most = col_launch_smem<NFFT, kFwdCols>(0, 1);
    if ((e = smem(fft_cols_tma_kernel<NFFT, kFwdCols>, most))) return e;
    if ((e = smem(fft_cols_multi_kernel<NFFT, kFwdCols>, most))) return e;
  }
  if (col_smem<NFFT, kAdjCols>() <= room) {
    const size_t most = col_launch_smem<NFFT, kAdjCols>(0, 1);
    if ((e = smem(fft_cols_tma_kernel<NFFT, kAdjCols>, most))) return e;
    if ((e = smem(fft_cols_multi_kernel<NFFT, kAdjCols>, most))) return e;
  }
  const int fsm = (int)fused_smem<NFFT>(NFFT / 2);
  if ((e = cudaFuncSetAttribute(fused_rows_multi_kernel<NFFT>, cudaFuncAttributeMaxDynamicSharedMemorySize, fsm)))
    return e;
  if ((e = cudaFuncSetAttribute(fused_rows_kernel<NFFT, kRowUpdateFwd>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                fsm)))
    return e;
  if ((e = cudaFuncSetAttribute(fused_rows_kernel<NFFT, kRowUpdate>, cudaFuncAttributeMaxDynamicSharedMemorySize, fsm)))
    return e;
  if constexpr (row_grad_size(NFFT))
    if ((e = smem(fused_rows_kernel<NFFT, kRowGrad>, (size_t)fsm))) return e;
  if constexpr (fused_ws_fits<NFFT>()) {
    if (fused_ws_smem<NFFT>() <= (size_t)optin - 1024) {
      const int wsm = (int)fused_ws_smem<NFFT>();
      if ((e = cudaFuncSetAttribute(fused_rows_ws_kernel<NFFT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    wsm)))
        return e;
      if ((e = cudaFuncSetAttribute(fused_rows_ws_kernel<NFFT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    wsm)))
        return e;
    }
  }
  return cudaSuccess;
}

#define PROP_FFT_SIZES(X) X(16) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512) X(768) X(1024)

cudaError_t dispatch(int n, int kind, const FftArgs& a, dim3 grid, int sms, cudaStream_t s) {
  switch (n) {
#define CASE(v) \
  case v: return launch<v>(kind, a, grid, sms, s);
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}

template <int NFFT>
cudaError_t launch_cols_tma(int kind, const CUtensorMap& tm, const ColArgs& a, int sms, cudaStream_t s) {
  const int per_sm = kind == kFwdCols ? col_ctas_per_sm<NFFT, kFwdCols>() : col_ctas_per_sm<NFFT, kAdjCols>();
  const int ctas = std::max(1, std::min(a.ntiles, per_sm * sms));
  const dim3 grid((unsigned)ctas), block(Shape<NFFT, kValsCols<NFFT>>::THREADS);
  if (kind == kFwdCols)
    return launch_dep(fft_cols_tma_kernel<NFFT, kFwdCols>, grid, block, col_launch_smem<NFFT, kFwdCols>(ctas, a.ntiles), s,
                      tm, a);
  return launch_dep(fft_cols_tma_kernel<NFFT, kAdjCols>, grid, block, col_launch_smem<NFFT, kAdjCols>(ctas, a.ntiles), s,
                    tm, a);
}

size_t cols_smem(int n, int kind) {
  switch (n) {
#define CASE(v) \
  case v: return kind == kFwdCols ? col_smem<v, kFwdCols>() : col_smem<v, kAdjCols>();
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return (size_t)1 << 30;
  }
}

int cols_per_sm(int n, int kind) {
  switch (n) {
#define CASE(v) \
  case v: return kind == kFwdCols ? col_ctas_per_sm<v, kFwdCols>() : col_ctas_per_sm<v, kAdjCols>();
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return 1;
  }
}

cudaError_t dispatch_cols_tma(int n, int kind, const CUtensorMap& tm, const ColArgs& a, int sms, cudaStream_t s) {
  switch (n) {
#define CASE(v) \
  case v: return launch_cols_tma<v>(kind, tm, a, sms, s);
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}

template <int NFFT>
cudaError_t launch_cols_multi(int kind, const MultiCols& m, int ctas, cudaStream_t s) {
  const dim3 grid((unsigned)ctas), block(Shape<NFFT, kValsCols<NFFT>>::THREADS);
  int ntiles = 0;
  for (int r = 0; r < m.nreq; ++r) ntiles += m.a[r].ntiles;
  if (kind == kFwdCols)
    return launch_dep(fft_cols_multi_kernel<NFFT, kFwdCols>, grid, block, col_launch_smem<NFFT, kFwdCols>(ctas, ntiles), s, m);
  return launch_dep(fft_cols_multi_kernel<NFFT, kAdjCols>, grid, block, col_launch_smem<NFFT, kAdjCols>(ctas, ntiles), s, m);
}

cudaError_t dispatch_cols_multi(int n, int kind, const MultiCols& m, int ctas, cudaStream_t s) {
  switch (n) {
#define CASE(v) \
  case v: return launch_cols_multi<v>(kind, m, ctas, s);
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t dispatch_fused_multi(int n, const MultiFused& m, cudaStream_t s) {
  switch (n) {
#define CASE(v) \
  case v: return launch_fused_multi<v>(m, s);
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}

// Largest power of two <= 256 dividing h (the tensor copy's box height).
int box_rows(int h) {
  int b = 256;
  while (b > 1 && h % b != 0) b >>= 1;
  return b;
}

// Box height of a column pass's input copies: where the adjoint skips unused
// blocks about a sixteenth of the column, a whole number of blocks (lower
// boxes skip more and cost more requests).
int col_box_rows(const Plan& p, int kind) {
  if (kind == kFwdCols) return box_rows(p.N);
  if (!p.grid_used || !p.grid_sparse) return box_rows(p.n);
  int bh = kGridBlock;
  while (bh * 16 < p.n) bh *= 2;
  return p.n % bh == 0 ? bh : kGridBlock;
}

// log2 of the 16-line tiles in two grid columns (bin strides 8, 16, 32, 64).
int used_shift(const Plan& p) {
  int s = 0;
  while ((kFftCols << s) < 2 * p.cs) ++s;
  return s;
}

ColArgs col_args(const Plan& p, int kind) {
  ColArgs a{};
  a.dst = kind == kFwdCols ? p.grid : p.rows;
  a.twiddle = p.twiddle;
  a.err = p.status_dev;
  a.nq = (size_t)p.n * p.cs;
  a.qtiles = (int)(a.nq / kFftCols);
  a.ntiles = a.qtiles * p.T;
  a.bh = col_box_rows(p, kind);
  a.nbox = (kind == kFwdCols ? p.N : p.n) / a.bh;
  a.used = p.grid_used;
  a.ushift = used_shift(p);
  a.box_mask = a.bh >= 64 * kGridBlock ? ~0ull : (1ull << std::max(1, a.bh / kGridBlock)) - 1;
  return a;
}

cudaError_t dispatch_fused(int n, const FusedArgs& a, int mode, dim3 grid, cudaStream_t s) {
  switch (n) {
#define CASE(v) \
  case v: return launch_fused<v>(a, mode, grid, s);
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}

// --- Centred unitary 2-D DFT of one N x N image (projection model) ----------
//
// Four passes of NFFT = N point transforms, kCartCols lines per CTA: forward rows,
// forward columns (scale 1/N; optionally masked), inverse columns (input
// optionally masked), inverse rows (scale 1/N); in a reconstruction both column
// passes and the blade's data term between them are one kernel.  The centring (image index i = x + N/2, k index u = N k + N/2) is
// the index map position -> (position + N/2) mod N on every input and
// output, which is where an unshifted DFT's position 0 holds x = 0 / k = 0.
struct CartArgs {
  const float2* src;
  float2* dst;
  const float2* twiddle;  // [N] exp(-2 pi i m / N)
  const uint8_t* mask;    // [N][N] blade support, or null
  const float2* y;        // data term: [N][N] k-space data of the blade
  const float2* yimg;     // data term: [N][N] DFT of the blade's image, or null (= y)
  float wk, wi;
  double* partials;
  unsigned int* counter;
  const double* loss_const;
  double* loss_out;
  int N;
  float scale;
};

__device__ __forceinline__ int cshift(int p, int N) {
  const int q = p + (N >> 1);
  return q >= N ? q - N : q;
}
// Lines are the rows r0 + col (elements contiguous).
struct InCartRows {
  const float2* src;
  int N;
  size_t r0;
  __device__ float2 operator()(int pos, int col) const { return src[(r0 + col) * N + cshift(pos, N)]; }
};
struct OutCartRows {
  float2* dst;
  int N;
  size_t r0;
  float scale;
  __device__ void operator()(int q, int col, float2 v) const { dst[(r0 + col) * N + cshift(q, N)] = cscale(v, scale); }
};
// Lines are the columns c0 + col (elements N apart).
struct InCartCols {
  const float2* src;
  const uint8_t* mask;
  int N, c0;
  __device__ float2 operator()(int pos, int col) const {
    const size_t i = (size_t)cshift(pos, N) * N + c0 + col;
    if (mask && !mask[i]) return make_float2(0.f, 0.f);
    return src[i];
  }
};
struct OutCartCols {
  float2* dst;
  const uint8_t* mask;
  int N, c0;
  float scale;
  __device__ void operator()(int q, int col, float2 v) const {
    const size_t i = (size_t)cshift(q, N) * N + c0 + col;
    float2 z = cscale(v, scale);
    if (mask && !mask[i]) z = make_float2(0.f, 0.f);
    dst[i] = z;
  }
};
// Forward column output of the data term: on the mask, r_k = Z - y,
// r_i = Z - yimg (the image term through the unitary DFT), loss += wk |r_k|^2 +
// wi |r_i|^2, and the gradient 2 (wk r_k + wi r_i), 0 elsewhere, into the CTA's
// buffer g[k position][col].  The data are loaded whether on the mask or not,
// so that no load waits for another.
struct OutCartLoss {
  float2* g;
  const uint8_t* mask;
  const float2* y;
  const float2* yimg;
  float wk, wi;
  int N, c0;
  float scale;
  float* acc;
  __device__ void operator()(int q, int col, float2 v) const {
    const int i = cshift(q, N) * N + c0 + col;
    const bool on = __ldg(&mask[i]) != 0;
    const float2 yy = __ldg(&y[i]);
    const float2 yi = yimg ? __ldg(&yimg[i]) : yy;
    const float2 z = cscale(v, scale);
    const float2 rk = make_float2(z.x - yy.x, z.y - yy.y);
    const float2 ri = make_float2(z.x - yi.x, z.y - yi.y);
    if (on) *acc += wk * fmaf(rk.x, rk.x, rk.y * rk.y) + wi * fmaf(ri.x, ri.x, ri.y * ri.y);
    g[q * kCartCols + col] = on ? make_float2(2.f * fmaf(wk, rk.x, wi * ri.x), 2.f * fmaf(wk, rk.y, wi * ri.y))
                                : make_float2(0.f, 0.f);
  }
};
struct InCartBuf {
  const float2* g;
  __device__ float2 operator()(int pos, int col) const { return g[pos * kCartCols + col]; }
};

template <int NFFT>
constexpr int cart_threads() {
  return NFFT / kValsCart<NFFT> * kCartCols;
}
template <int NFFT>
constexpr size_t cart_smem() {
  return (size_t)NFFT * kCartCols * sizeof(float2) + (size_t)Shape<NFFT, kValsCart<NFFT>>::TW * sizeof(float2);
}
template <int NFFT>
constexpr size_t cart_loss_smem() {  // and the gradient between the two column passes
  return cart_smem<NFFT>() + (size_t)NFFT * kCartCols * sizeof(float2);
}

template <int NFFT, int PASS>
__global__ void __launch_bounds__(cart_threads<NFFT>()) cart_fft_kernel(CartArgs a) {
  constexpr int EV = kValsCart<NFFT>;
  constexpr int CC = kCartCols;
  extern __shared__ float2 smem[];
  float2* X = smem;
  float2* tw = smem + NFFT * CC;
  build_twiddles<NFFT, EV>(tw, a.twiddle);
  grid_dep_wait();
  grid_dep_release();
  __syncthreads();
  const int col = threadIdx.x % CC;
  const int tl = threadIdx.x / CC;
  const int l0 = blockIdx.x * CC;
  if constexpr (PASS == kCartRowsFwd) {
    InCartRows in{a.src, NFFT, (size_t)l0};
    OutCartRows out{a.dst, NFFT, (size_t)l0, a.scale};
    fft_pass<NFFT, EV, -1, 0, 1, false, false, CtaSync, InCartRows, OutCartRows, NoHook, CC>(X, tw, col, tl, in, out);
  } else if constexpr (PASS == kCartColsFwd) {
    InCartCols in{a.src, nullptr, NFFT, l0};
    OutCartCols out{a.dst, a.mask, NFFT, l0, a.scale};
    fft_pass<NFFT, EV, -1, 0, 1, false, false, CtaSync, InCartCols, OutCartCols, NoHook, CC>(X, tw, col, tl, in, out);
  } else if constexpr (PASS == kCartColsLoss) {
    float2* g = tw + Shape<NFFT, EV>::TW;
    InCartCols in{a.src, nullptr, NFFT, l0};
    float acc = 0.f;
    OutCartLoss mid{g, a.mask, a.y, a.yimg, a.wk, a.wi, NFFT, l0, a.scale, &acc};
    fft_pass<NFFT, EV, -1, 0, 1, false, false, CtaSync, InCartCols, OutCartLoss, NoHook, CC>(X, tw, col, tl, in, mid);
    __syncthreads();
    InCartBuf back{g};
    OutCartCols out{a.dst, nullptr, NFFT, l0, 1.f};
    fft_pass<NFFT, EV, +1, 0, 1, false, false, CtaSync, InCartBuf, OutCartCols, NoHook, CC>(X, tw, col, tl, back, out);
    finish_loss(acc, a.partials, a.counter, a.loss_const, a.loss_out);
  } else if constexpr (PASS == kCartColsInv) {
    InCartCols in{a.src, a.mask, NFFT, l0};
    OutCartCols out{a.dst, nullptr, NFFT, l0, a.scale};
    fft_pass<NFFT, EV, +1, 0, 1, false, false, CtaSync, InCartCols, OutCartCols, NoHook, CC>(X, tw, col, tl, in, out);
  } else {
    InCartRows in{a.src, NFFT, (size_t)l0};
    OutCartRows out{a.dst, NFFT, (size_t)l0, a.scale};
    fft_pass<NFFT, EV, +1, 0, 1, false, false, CtaSync, InCartRows, OutCartRows, NoHook, CC>(X, tw, col, tl, in, out);
  }
}

template <int NFFT>
cudaError_t launch_cart(int pass, const CartArgs& a, cudaStream_t s) {
  const dim3 grid(NFFT / kCartCols), block(cart_threads<NFFT>());
  const size_t smem = cart_smem<NFFT>();
  switch (pass) {
    case kCartRowsFwd: return launch_dep(cart_fft_kernel<NFFT, kCartRowsFwd>, grid, block, smem, s, a);
    case kCartColsFwd: return launch_dep(cart_fft_kernel<NFFT, kCartColsFwd>, grid, block, smem, s, a);
    case kCartColsInv: return launch_dep(cart_fft_kernel<NFFT, kCartColsInv>, grid, block, smem, s, a);
    case kCartColsLoss: return launch_dep(cart_fft_kernel<NFFT, kCartColsLoss>, grid, block, cart_loss_smem<NFFT>(), s, a);
    default: return launch_dep(cart_fft_kernel<NFFT, kCartRowsInv>, grid, block, smem, s, a);
  }
}

template <int NFFT>
cudaError_t configure_cart() {
  const int smem = (int)cart_smem<NFFT>();
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(cart_fft_kernel<NFFT, kCartRowsFwd>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)))
    return e;
  if ((e = cudaFuncSetAttribute(cart_fft_kernel<NFFT, kCartColsFwd>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)))
    return e;
  if ((e = cudaFuncSetAttribute(cart_fft_kernel<NFFT, kCartColsInv>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)))
    return e;
  if ((e = cudaFuncSetAttribute(cart_fft_kernel<NFFT, kCartColsLoss>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)cart_loss_smem<NFFT>())))
    return e;
  return cudaFuncSetAttribute(cart_fft_kernel<NFFT, kCartRowsInv>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

cudaError_t dispatch_fused_ws(int n, const CUtensorMap& tm, const FusedArgs& a, bool fwd_tail, int ctas,
                              cudaStream_t s) {
  switch (n) {
#define CASE(v) \
  case v: return launch_fused_ws<v>(tm, a, fwd_tail, ctas, s);
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}

// Whether the warp-specialised row kernel can run: its shared memory fits, and
// where its two groups share out the launch's registers, the launch has the 64
// a thread that the split hands out (it would wait forever for registers that
// it does not have).  The per-row kernel serves what it cannot.
template <int NFFT>
bool fused_ws_runs_n(size_t room) {
  if constexpr (fused_ws_fits<NFFT>()) {
    if (fused_ws_smem<NFFT>() > room) return false;
    if (Shape<NFFT, kValsFused<NFFT>>::THREADS != kUpdThreads) return true;
    cudaFuncAttributes fa, fb;
    if (cudaFuncGetAttributes(&fa, fused_rows_ws_kernel<NFFT, true>) != cudaSuccess ||
        cudaFuncGetAttributes(&fb, fused_rows_ws_kernel<NFFT, false>) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    return fa.numRegs >= 64 && fb.numRegs >= 64;
  }
  return false;
}

bool fused_ws_runs(int n, size_t room) {
  switch (n) {
#define CASE(v) \
  case v: return fused_ws_runs_n<v>(room);
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return false;
  }
}

FftArgs base_args(const Plan& p) {
  FftArgs a{};
  a.deapod = p.deapod;
  a.twiddle = p.twiddle;
  a.Nf = p.Nf;
  a.C = p.cs;
  a.Cv = p.chunk;
  a.f0 = 0;
  a.scale = 1.f;
  a.used = p.grid_used;
  a.ushift = used_shift(p);
  return a;
}

}  // namespace

cudaError_t fft_configure(int n) {
  switch (n) {
#define CASE(v) \
  case v: return configure_n<v>();
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t fft_forward_rows(const Plan& p, const float2* V, int f0, cudaStream_t s) {
  FftArgs a = base_args(p);
  a.src = V;
  a.dst = p.rows;
  a.f0 = f0;
  a.Cv = std::min(p.chunk, p.Nf - f0);
  dim3 grid(a.C, p.T * p.N);  // x: lines
  return dispatch(p.n, kFwdRows, a, grid, p.num_sms, s);
}

void fft_make_maps(Plan& p) {
  p.cols_tma_fwd = p.cols_tma_adj = false;
  using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static EncodeFn encode = nullptr;
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
      cudaGetLastError();
      return;
    }
    encode = reinterpret_cast<EncodeFn>(fn);
  }
  if (p.cs % 2 != 0 || p.T > 65536) return;
  const size_t nq = (size_t)p.n * p.cs;
  auto make = [&](CUtensorMap* tm, float2* base, int h, int bh) {
    const cuuint64_t dims[3] = {(cuuint64_t)(2 * nq), (cuuint64_t)h, (cuuint64_t)p.T};
    const cuuint64_t strides[2] = {(cuuint64_t)(2 * nq * sizeof(float)), (cuuint64_t)(2 * nq * h * sizeof(float))};
    const cuuint32_t box[3] = {(cuuint32_t)(2 * kFftCols), (cuuint32_t)bh, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    return encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  const size_t room = (size_t)p.smem_optin - 1024;
  p.cols_tma_fwd = cols_smem(p.n, kFwdCols) <= room && make(&p.tm_rows, p.rows, p.N, col_box_rows(p, kFwdCols));
  p.cols_tma_adj = cols_smem(p.n, kAdjCols) <= room && make(&p.tm_grid, p.grid, p.n, col_box_rows(p, kAdjCols));
  // fused row kernel input: [T N][n][2 cs] floats, box = 16 bins x box_rows(n) positions of one row.
  // Automatic choice: the warp-specialised kernel pipelines the units of a
  // CTA, which pays off once every SM has several (at 3.4 units per SM the
  // per-row CTAs were faster, at 27 the warp-specialised kernel by a fifth).
  p.fused_ws = false;
  const long units = (long)((p.Nf + kFftCols - 1) / kFftCols) * p.T * p.N;
  const bool want = p.row_kernel == 2 || (p.row_kernel == 0 && units >= 8L * p.num_sms);
  if (want && p.cs % kFftCols == 0 && p.nchunks == 1 && (size_t)p.T * p.N <= 0xffffffffu &&
      fused_ws_runs(p.n, room)) {
    const cuuint64_t dims[3] = {(cuuint64_t)(2 * p.cs), (cuuint64_t)p.n, (cuuint64_t)p.T * p.N};
    const cuuint64_t strides[2] = {(cuuint64_t)(2 * p.cs * sizeof(float)),
                                   (cuuint64_t)(2 * (size_t)p.cs * p.n * sizeof(float))};
    const cuuint32_t box[3] = {(cuuint32_t)(2 * kFftCols), (cuuint32_t)box_rows(p.n), 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    p.fused_ws = encode(&p.tm_fused, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, p.rows, dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  }
}

cudaError_t fft_forward_cols(const Plan& p, cudaStream_t s) {
  if (p.cols_tma_fwd) return dispatch_cols_tma(p.n, kFwdCols, p.tm_rows, col_args(p, kFwdCols), p.num_sms, s);
  FftArgs a = base_args(p);
  a.src = p.rows;
  a.dst = p.grid;
  dim3 grid(p.n * p.cs, p.T);  // x: lines
  return dispatch(p.n, kFwdCols, a, grid, p.num_sms, s);
}

cudaError_t fft_adjoint_cols(const Plan& p, cudaStream_t s) {
  if (p.cols_tma_adj) return dispatch_cols_tma(p.n, kAdjCols, p.tm_grid, col_args(p, kAdjCols), p.num_sms, s);
  FftArgs a = base_args(p);
  a.src = p.grid;
  a.dst = p.rows;
  dim3 grid(p.n * p.cs, p.T);  // x: lines
  return dispatch(p.n, kAdjCols, a, grid, p.num_sms, s);
}

cudaError_t fft_adjoint_rows(const Plan& p, float2* out, int f0, float scale, cudaStream_t s) {
  FftArgs a = base_args(p);
  a.src = p.rows;
  a.dst = out;
  a.f0 = f0;
  a.scale = scale;
  a.Cv = std::min(p.chunk, p.Nf - f0);
  dim3 grid(a.Cv, p.T * p.N);  // x: lines
  return dispatch(p.n, kAdjRows, a, grid, p.num_sms, s);
}

namespace {
FusedArgs fused_args(const Plan& p, const float2* Vin, float2* m, float2* v, float2* Vout, const AdamArgs& aa,
                     const Reducer* red, const double* data_loss, double* loss_out) {
  FusedArgs a{};
  a.rows = p.rows;
  a.deapod = p.deapod;
  a.twiddle = p.twiddle;
  a.Vin = Vin;
  a.Vout = Vout;
  a.m = m;
  a.v = v;
  a.partials = red->partials;
  a.counter = red->counter;
  a.data_loss = data_loss;
  a.loss_out = loss_out;
  a.N = p.N;
  a.Nf = p.Nf;
  a.C = p.cs;
  a.T = p.T;
  a.scale = 1.0f / (float)p.N;
  a.ad = aa;
  a.err = p.status_dev;
  a.nfb = (p.Nf + kFftCols - 1) / kFftCols;
  a.units = a.nfb * p.T * p.N;
  return a;
}

// Column pass over a batch: CTAs split by tile count.
cudaError_t cols_batch(Plan* const* ps, int count, int kind, cudaStream_t s) {
  if (count < 1 || count > kMaxBatch) return cudaErrorInvalidValue;
  bool tma = true;
  for (int r = 0; r < count; ++r) {
    tma = tma && (kind == kFwdCols ? ps[r]->cols_tma_fwd : ps[r]->cols_tma_adj);
    if (ps[r]->n != ps[0]->n) return cudaErrorInvalidValue;
  }
  if (!tma) {  // untiled fallback: one launch per plan
    for (int r = 0; r < count; ++r) {
      const cudaError_t e = kind == kFwdCols ? fft_forward_cols(*ps[r], s) : fft_adjoint_cols(*ps[r], s);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  MultiCols m{};
  m.nreq = count;
  long work[kMaxBatch];
  int cap[kMaxBatch];
  for (int r = 0; r < count; ++r) {
    m.tm[r] = kind == kFwdCols ? ps[r]->tm_rows : ps[r]->tm_grid;
    m.a[r] = col_args(*ps[r], kind);
    work[r] = m.a[r].ntiles;
    cap[r] = std::max(1, m.a[r].ntiles);
  }
  const int per_sm = cols_per_sm(ps[0]->n, kind);
  const int ctas = split_ctas(work, cap, count, std::max(count, per_sm * ps[0]->num_sms), m.cta_begin);
  return dispatch_cols_multi(ps[0]->n, kind, m, ctas, s);
}
}  // namespace

cudaError_t fft_forward_cols_batch(Plan* const* ps, int count, cudaStream_t s) {
  return cols_batch(ps, count, kFwdCols, s);
}
cudaError_t fft_adjoint_cols_batch(Plan* const* ps, int count, cudaStream_t s) {
  return cols_batch(ps, count, kAdjCols, s);
}

cudaError_t fused_rows_update_batch(const BatchIter* it, int count, cudaStream_t s) {
  if (count < 1 || count > kMaxBatch) return cudaErrorInvalidValue;
  MultiFused m{};
  m.nreq = 0;
  m.unit_begin[0] = 0;
  for (int r = 0; r < count; ++r) {
    const Plan& p = *it[r].p;
    if (p.nchunks != 1 || p.n != it[0].p->n) return cudaErrorInvalidValue;
    if (p.fused_ws) {  // the persistent warp-specialised kernel runs on its own
      const cudaError_t e = fused_rows_update(p, it[r].Vin, p.adam_m, p.adam_v, it[r].Vout, it[r].aa, &p.red_tv,
                                              p.scalars, it[r].loss_out, it[r].fwd_tail, s);
      if (e != cudaSuccess) return e;
      continue;
    }
    const int q = m.nreq++;
    m.a[q] = fused_args(p, it[r].Vin, p.adam_m, p.adam_v, it[r].Vout, it[r].aa, &p.red_tv, p.scalars,
                        it[r].loss_out);
    if (m.a[q].units > p.red_tv.capacity) return cudaErrorInvalidValue;
    m.fwd_tail[q] = it[r].fwd_tail ? 1 : 0;
    m.unit_begin[q + 1] = m.unit_begin[q] + m.a[q].units;
  }
  if (m.nreq == 0) return cudaSuccess;
  return dispatch_fused_multi(it[0].p->n, m, s);
}

cudaError_t fused_rows_update(const Plan& p, const float2* Vin, float2* m, float2* v, float2* Vout,
                              const AdamArgs& aa, const Reducer* red, const double* data_loss, double* loss_out,
                              bool fwd_tail, cudaStream_t s) {
  if (p.nchunks != 1 || !red) return cudaErrorInvalidValue;
  FusedArgs a = fused_args(p, Vin, m, v, Vout, aa, red, data_loss, loss_out);
  if (p.fused_ws) {
    a.bh = box_rows(p.n);
    a.nbox = p.n / a.bh;
    const int ctas = std::max(1, std::min(a.units, p.num_sms));
    if (ctas > red->capacity) return cudaErrorInvalidValue;
    return dispatch_fused_ws(p.n, p.tm_fused, a, fwd_tail, ctas, s);
  }
  if (a.units > red->capacity) return cudaErrorInvalidValue;
  return dispatch_fused(p.n, a, fwd_tail ? kRowUpdateFwd : kRowUpdate, dim3(a.nfb, p.T * p.N), s);
}

// Whether the gradient of the loss is taken by the fused row kernel or by the
// adjoint row pass and the TV kernel (the same values; whole prop_loss_grad
// calls, separate -> fused).  Fused saves a launch and the gradient's trip
// through memory: 3 to 10 % of a call (one frame of 64^2 x 32 bins 0.91x, 256^2 x
// 16 bins x 8 frames 0.90x).  But the lanes of a missing bin run along, so with
// few bins and several frames it loses (512^2 x 1 bin x 32 frames: 395 us
// separate, 1520 fused, of these passes; 192^2 x 5 bins x 32 frames 1.09x a
// call); below N = 32 its CTAs are a warp or two (16^2 x 64 bins x 32 frames 108
// against 119 us a call), and at 512 one fits an SM.
bool fused_rows_grad_pays(const Plan& p) {
  if (p.nchunks != 1 || !row_grad_size(p.n)) return false;
  if (p.T == 1) return p.N <= 256 || p.Nf > 2;
  if (p.N <= 32) return p.N == 32 && p.Nf >= 5 && p.Nf <= kFftCols;
  return p.Nf >= (p.N <= 128 ? 5 : 12);
}

cudaError_t fused_rows_grad(const Plan& p, const float2* V, float2* grad, const AdamArgs& aa, const Reducer* red,
                            const double* data_loss, double* loss_out, cudaStream_t s) {
  if (p.nchunks != 1 || !red) return cudaErrorInvalidValue;
  const FusedArgs a = fused_args(p, V, nullptr, nullptr, grad, aa, red, data_loss, loss_out);
  if (a.units > red->capacity) return cudaErrorInvalidValue;
  return dispatch_fused(p.n, a, kRowGrad, dim3(a.nfb, p.T * p.N), s);
}

cudaError_t cart_fft_configure(int N) {
  switch (N) {
#define CASE(v) \
  case v: return configure_cart<v>();
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t cart_fft_pass(int N, int pass, const float2* src, float2* dst, const float2* twiddleN,
                          const uint8_t* mask, const CartLoss* loss, float scale, cudaStream_t s) {
  CartArgs a{};
  a.src = src;
  a.dst = dst;
  a.twiddle = twiddleN;
  a.mask = mask;
  a.N = N;
  a.scale = scale;
  if ((pass == kCartColsLoss) != (loss != nullptr)) return cudaErrorInvalidValue;
  if (loss) {
    if (!loss->red || !mask || loss->red->capacity < N / kCartCols) return cudaErrorInvalidValue;
    a.y = loss->y;
    a.yimg = loss->yimg;
    a.wk = loss->wk;
    a.wi = loss->wi;
    a.partials = loss->red->partials;
    a.counter = loss->red->counter;
    a.loss_const = loss->loss_const;
    a.loss_out = loss->loss_out;
  }
  switch (N) {
#define CASE(v) \
  case v: return launch_cart<v>(pass, a, s);
    PROP_FFT_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace prop
