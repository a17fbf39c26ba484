// Time transform by FFT (Methods, "Workflow Architecture": psi~(k, w) = F_t[psi(k, t) - <psi(k, t)>_t],
// I(k, w) = |psi~|^2) in one pass over the exit-wave stack, in FP32.
//
// A CTA takes C neighbouring q columns of one probe and all F frames: it loads them once (T threads
// a column, E frames a thread, the engine of fft.cuh), removes the mean, transforms along the frames
// through shared memory and stores |psi~|^2, or its sum over the columns (the spectrum image), or
// psi~ itself (one process's share of a frame-sharded transform).  The stack is read once and the
// result written once; the dense forms of the transform read it two or three times, write a
// residual or split operands and do O(F) work per element where this does O(log F).  1024 frames x
// 65536 q: 14.6 ms dense FP32, 0.24 ms here (3.3 TB/s); a partial transform of 256 of 512 frames: 2.14 ms,
// 0.17 ms.  The image at 256 frames is bound by latency and the FP32 pipe (pipe 61% busy, 59% of the issue slots
// by 22 warps, shared memory 44%, DRAM 40%), the forms of 1024 points by latency at the 8 warps that hold
// them in registers (pipe 44%, issue 40%, DRAM 40%; chirp-z 44%, 49%, 14%).
//
// Mean to FP64-class precision, as the dense forms have it: a column is summed as FP32 pairs (error-free
// two-sums, in the thread, over the lanes and over the warps).  Every frame loses the mean rounded to float,
// one subtraction with one rounding; what the rounded mean leaves of the column's sum, F times half a last
// place at most, is the same in every frame, so it reaches bin 0 alone and is taken out of it there.  Columns
// that do not change give exactly zero.  Plain FP32 sums of psi_n - psi_0 are faster (1024 frames x 65536 q
// 235 us, 243 now; image of 32 probes at 256 frames 435, 463; 501 frames 315, 330), but round the residual
// twice, and their own error came back F-fold in bin 0: up to 15 times the rounding of the sum itself in
// columns whose first frame stands out.  Forming the residual exactly against a mean of two floats gave the
// same and took longer (266, 521 and 346 us).
//
// Frame counts: the engine's own lengths directly; any other F up to 2048 by Bluestein's chirp-z
// identity m n = (m^2 + n^2 - (m - n)^2) / 2, as a cyclic convolution of length M >= 2 F - 1 with a
// precomputed chirp spectrum (two transforms of length M; the final chirp has modulus 1 and is left
// out where only |psi~|^2 is wanted).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "fft.cuh"
#include "tacaw_api_internal.h"

namespace tacaw {

enum TimeOut { TIME_S, TIME_DETECTOR, TIME_TILDE };

// Shape of a kernel: elements per thread, columns per CTA, CTAs per SM, and whether a thread loads its
// next column while it transforms this one.  Per length the fastest of 4 to 14 shapes on one GB300
// (ps per element of the stack; one shape for all uses -> these, before the mean was summed in pairs): 256
// points S 3.21 -> 2.95, image 3.05 -> 2.85, chirp-z 7.64 -> 7.08; 512: S 4.99 -> 3.39, image 4.88 -> 3.14,
// chirp-z 11.4 -> 8.0; 1024: S 7.02 -> 4.95, image 5.41 -> 4.42, chirp-z 13.0 -> 11.2; 2048: S 7.91 -> 7.54,
// image 7.43 -> 5.87, chirp-z 19.8 -> 14.9; 4096: chirp-z 27.7 -> 16.9.  Now S, image, chirp-z S at 256 points
// 3.00, 2.73, 7.17; 512: 3.49, 2.86, 8.14; 1024: 4.95, 4.11, 10.7; 2048: 7.54, 5.46, 14.9.  16 columns are whole
// 128-byte lines of the stack; more columns of the long transforms would leave one CTA per SM.
struct TimeShape {
  int e, c, minb;
  bool prefetch;
};
constexpr TimeShape time_shape(int n, int out, bool chirp) {
  switch (n) {
    case 32: return {8, 32, 4, !chirp};
    case 64: return {8, 32, 2, !chirp};
    case 96: return {24, 32, 2, false};
    case 128: return {16, 32, 2, !chirp};
    case 192: return {24, 16, 2, false};
    case 256: return chirp ? TimeShape{16, 8, 4, false} : TimeShape{16, 16, out == TIME_DETECTOR ? 3 : 2, true};
    case 384: return {24, 16, 1, false};
    case 512: return chirp || out == TIME_DETECTOR ? TimeShape{32, 8, 3, false} : TimeShape{32, 16, 1, true};
    case 768: return {24, 8, 1, false};
    case 1024: return {32, 8, !chirp && out == TIME_DETECTOR ? 2 : 1, !chirp};
    case 1152: return {24, 8, 1, false};
    case 2048:
      return chirp || out == TIME_DETECTOR ? TimeShape{32, 4, 1, false}
             : out == TIME_S               ? TimeShape{16, 4, 1, true}
                                           : TimeShape{32, 8, 1, false};
    default: return {32, 2, 1, false};
  }
}
template <int N, int OUT, bool BLUE>
struct TimeCfg {
  static constexpr TimeShape SHAPE = time_shape(N, OUT, BLUE);
  static constexpr int E = SHAPE.e, T = N / E, C = SHAPE.c, THREADS = T * C, MINB = SHAPE.minb;
  static constexpr int SH = E == 32 ? 5 : 0;
  static constexpr int SCRATCH = (N + (SH ? N >> SH : 0)) * C * (int)sizeof(float2), TILE = N * C * (int)sizeof(float2);
  // The next tile comes into registers where they are free.  The spectrum image keeps its running sums
  // in them and the chirp-z forms need them; there it comes by cp.async into shared memory (each thread
  // copies and reads its own elements) for the short transforms and for S through 1024 points: ps an
  // element without -> with it, image and chirp-z S at 32 points 3.53 -> 3.25 and 9.49 -> 7.33, 128
  // points 3.06 -> 2.73 and 7.57 -> 6.95, chirp-z S at 1024 11.2 -> 10.1.  At 256 and 512 points the
  // second buffer costs more than it gives (image 2.72 -> 2.89 and 3.29 -> 5.26).
  static constexpr bool ASYNC = (OUT == TIME_DETECTOR || BLUE) && (N <= 128 || (N == 1024 && OUT != TIME_DETECTOR));
  static constexpr bool PREFETCH = SHAPE.prefetch && OUT != TIME_DETECTOR && !BLUE;
  static constexpr int SMEM = SCRATCH + (ASYNC ? TILE : 0);
};

struct TimeArgs {
  const float2* psi;  // [P][nf][in_nq]
  const float2* ref;  // TIME_TILDE: [P][in_nq] static reference; else unused
  int64_t P, F, nf, f0;
  int64_t in_nq;
  const int32_t* in_qsel;
  int64_t nsel;
  int64_t out_nq;
  const int32_t* out_qsel;
  float* S;        // TIME_S: [P][F][out_nq]
  double* part;    // TIME_DETECTOR: [P][gridDim.x][F]
  float2* tilde;   // TIME_TILDE: [P][F][nsel]
  const float2* tw;     // FFT pass tables
  const float2* chirp;  // Bluestein: exp(-i pi n^2 / F), n < F
  const float2* bhat;   // Bluestein: spectrum of the conjugate chirp over M
  int tpc;              // column tiles per CTA
};

// Column tiles one CTA of the spectrum image adds up before it stores its partial sums.  Fixed, so
// that the order of the sums does not depend on how many probes a call holds.
constexpr int TIME_DET_TILES = 8;

// The sums over the C columns of a CTA, C neighbouring lanes of a warp: n bins a lane as FP32 pairs.  In
// each step two lanes O apart add theirs; while n is even each of the two keeps one half of the bins
// (from e0 on), then both keep all and one of them writes.  In FP64 (three operations an element on a
// pipe of two results a clock) these sums took a third of the pass at 256 frames.  Before the mean was summed
// in pairs too: image of 32 probes, 256 frames 465 -> 435 us, ps an element at 32, 192, 512, 2048 frames
// 3.23 -> 2.56, 3.52 -> 2.67, 3.17 -> 2.73, 5.88 -> 5.15.
__host__ __device__ constexpr int kept_bins(int n, int c) { return c == 1 ? n : kept_bins(n % 2 ? n : n / 2, c / 2); }
template <int n, int O>
__device__ __forceinline__ void column_pairs(float* hi, float* lo, int c, int& e0, bool& writer) {
  if constexpr (O > 0) {
    constexpr int KEEP = n % 2 ? n : n / 2;
    const bool up = c & O;
#pragma unroll
    for (int e = 0; e < KEEP; ++e) {
      const int other = n % 2 ? e : e + KEEP;
      const float h = up ? hi[other] : hi[e], l = up ? lo[other] : lo[e];
      const float gh = up ? hi[e] : hi[other], gl = up ? lo[e] : lo[other];
      float err;
      two_sum(h, __shfl_xor_sync(0xffffffffu, gh, O), hi[e], err);
      lo[e] = __fadd_rn(__fadd_rn(l, __shfl_xor_sync(0xffffffffu, gl, O)), err);
    }
    if (n % 2) writer = writer && !up;
    else if (up) e0 += KEEP;
    column_pairs<KEEP, O / 2>(hi, lo, c, e0, writer);
  }
}

// Complex FP32 pairs, both parts in packed instructions.
__device__ __forceinline__ float2 shfl_xor2(float2 a, int o) {
  return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
}
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
  s = a + b;
  const float2 bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
// (h, l) += (xh, xl)
__device__ __forceinline__ void pair_add2(float2& h, float2& l, float2 xh, float2 xl) {
  float2 e;
  two_sum2(h, xh, h, e);
  l = (l + xl) + e;
}
// The mean (h + l) / F rounded to float, and the rest of the sum, rest = h + l - F mean.  The remainder of
// a rounded quotient, h - F q, is exact (a few F units of q's last place), so a column of F equal
// frames has exactly that mean and no rest.
__device__ __forceinline__ void pair_mean2(float2 h, float2 l, float F, float inv, float2& mean, float2& rest) {
  const float2 q = inv * h;
  mean = fma2(inv, fma2(-F, q, h) + l, q);
  rest = fma2(-F, mean, h) + l;
}

template <int N, int OUT, bool BLUE>
__global__ void __launch_bounds__(TimeCfg<N, OUT, BLUE>::THREADS, TimeCfg<N, OUT, BLUE>::MINB)
    k_time_fft(const TimeArgs a) {
  grid_dependency_wait();
  using TC = TimeCfg<N, OUT, BLUE>;
  constexpr int E = TC::E, T = TC::T, C = TC::C, WARPS = TC::THREADS / 32;
  constexpr int IN = BLUE ? E / 2 : E;  // chirp-z: N >= 2 F - 1 is even, so t + T e < F only for e < E / 2
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int64_t p = blockIdx.y + (int64_t)gridDim.y * blockIdx.z;
  if (p >= a.P) return;
  const int c = threadIdx.x % C, t = threadIdx.x / C;
  const ColIdx<C, TC::SH> idx{c};
  const BlockSync sync;
  const int F = (int)a.F;
  const int64_t ntiles = (a.nsel + C - 1) / C;
  float hi[OUT == TIME_DETECTOR ? E : 1], lo[OUT == TIME_DETECTOR ? E : 1];
  if constexpr (OUT == TIME_DETECTOR) {
#pragma unroll
    for (int e = 0; e < E; ++e) hi[e] = lo[e] = 0.f;
  }
  const int64_t tile0 = (int64_t)blockIdx.x * a.tpc, tile1 = tile0 + a.tpc < ntiles ? tile0 + a.tpc : ntiles;
  // frames t + T e of column tile * C + c (zeros past the last one); x0: the static reference (TIME_TILDE)
  const auto load = [&](float2 (&u)[E], float2& x0, int64_t tile) {
    const int64_t j = tile * C + c, jj = j < a.nsel ? j : a.nsel - 1;  // past the end: the last one, unstored
    const int64_t q = a.in_qsel ? a.in_qsel[jj] : jj;
    if constexpr (OUT == TIME_TILDE) {
      const float2* col = a.psi + (size_t)p * a.nf * a.in_nq + q;
      x0 = a.ref[(size_t)p * a.in_nq + q];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int64_t n = t + T * e - a.f0;
        u[e] = n >= 0 && n < a.nf ? col[(size_t)n * a.in_nq] : x0;
      }
    } else {
      const float2* col = a.psi + (size_t)p * F * a.in_nq + q;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int n = t + T * e;
        u[e] = !BLUE || n < F ? col[(size_t)n * a.in_nq] : make_float2(0.f, 0.f);
      }
    }
  };
  // the same into this thread's slots of the tile buffer; x0 into a register
  float2* slots = reinterpret_cast<float2*>(smraw + TC::SCRATCH) + threadIdx.x;  // [E][THREADS]
  const auto fetch = [&](float2& x0, int64_t tile) {
    const int64_t j = tile * C + c, jj = j < a.nsel ? j : a.nsel - 1;
    const int64_t q = a.in_qsel ? a.in_qsel[jj] : jj;
    const bool part = OUT == TIME_TILDE;
    const float2* col = a.psi + (size_t)p * (part ? a.nf : (int64_t)F) * a.in_nq + q;
    if (part) x0 = a.ref[(size_t)p * a.in_nq + q];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int64_t n = t + T * e - (part ? a.f0 : 0);
      if (part ? n >= 0 && n < a.nf : !BLUE || n < F)
        cp_async8(slots + TC::THREADS * e, col + (size_t)n * a.in_nq);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const auto collect = [&](float2 (&u)[E], float2 x0) {
    cp_async_wait_all();
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int64_t n = t + T * e - (OUT == TIME_TILDE ? a.f0 : 0);
      const bool in = OUT == TIME_TILDE ? n >= 0 && n < a.nf : !BLUE || n < F;
      u[e] = in ? slots[TC::THREADS * e] : OUT == TIME_TILDE ? x0 : make_float2(0.f, 0.f);
    }
  };
  float2 v[E], x0 = make_float2(0.f, 0.f);
  if (TC::ASYNC) fetch(x0, tile0);
  else load(v, x0, tile0);
  for (int64_t tile = tile0; tile < tile1; ++tile) {
    const int64_t j = tile * C + c;
    const bool live = j < a.nsel;
    float2 next[E], next0 = x0, rest = make_float2(0.f, 0.f);
    if (TC::ASYNC) collect(v, x0);
    if (TC::PREFETCH && tile + 1 < tile1) load(next, next0, tile + 1);
    if constexpr (OUT == TIME_TILDE) {
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = v[e] - x0;
      if (TC::ASYNC) __syncthreads();  // every slot has been read
    } else {
      float2 hs = v[0], ls = make_float2(0.f, 0.f);
#pragma unroll
      for (int e = 1; e < IN; ++e) {
        float2 err;
        two_sum2(hs, v[e], hs, err);
        ls = ls + err;
      }
      // the column's sum: over the lanes of a warp that share it, then over the warps
#pragma unroll
      for (int o = C; o < 32; o <<= 1)
        pair_add2(hs, ls, shfl_xor2(hs, o), shfl_xor2(ls, o));
      float4* part = reinterpret_cast<float4*>(smraw);  // [WARPS][C]
      __syncthreads();  // the previous tile's readers of the scratch are done
      if ((threadIdx.x & 31) < C) part[(threadIdx.x >> 5) * C + c] = make_float4(hs.x, hs.y, ls.x, ls.y);
      __syncthreads();
      // the lanes of a column share the warps' sums, then add theirs
      constexpr int L = 32 / C < WARPS ? 32 / C : WARPS;
      static_assert(WARPS % L == 0, "every lane takes as many of the warps' sums");
      const int l0 = (threadIdx.x & 31) / C % L;
      float4 q = part[l0 * C + c];
      hs = make_float2(q.x, q.y);
      ls = make_float2(q.z, q.w);
#pragma unroll
      for (int w = L; w < WARPS; w += L) {
        q = part[(w + l0) * C + c];
        pair_add2(hs, ls, make_float2(q.x, q.y), make_float2(q.z, q.w));
      }
#pragma unroll
      for (int o = C; o < C * L; o <<= 1) pair_add2(hs, ls, shfl_xor2(hs, o), shfl_xor2(ls, o));
      float2 mean;
      pair_mean2(hs, ls, (float)F, 1.f / (float)F, mean, rest);
#pragma unroll
      for (int e = 0; e < E; ++e)
        v[e] = e < IN && (!BLUE || t + T * e < F) ? v[e] - mean : make_float2(0.f, 0.f);
    }
    // (both branches have passed a barrier after the slots were read)
    if (TC::ASYNC && tile + 1 < tile1) fetch(x0, tile + 1);
    if constexpr (BLUE) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int n = t + T * e;
        if (n < F) v[e] = cmul(v[e], __ldg(a.chirp + n));
      }
      fft<N, -1>(v, sm, idx, t, a.tw, sync);
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = cmul(v[e], __ldg(a.bhat + t + T * e));
      fft<N, +1>(v, sm, idx, t, a.tw, sync);
    } else {
      fft<N, -1>(v, sm, idx, t, a.tw, sync);
    }
    if (OUT != TIME_TILDE && t == 0) v[0] = v[0] - rest;
    if constexpr (OUT == TIME_DETECTOR) {
      if (live) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          // FP32 pair: the exact errors of at most TIME_DET_TILES sums add up in lo, so that with the lanes'
          // sums below a pair is off by less than 2^-43 of itself, 2^19 times less than the float returned
          float err;
          two_sum(hi[e], v[e].x * v[e].x + v[e].y * v[e].y, hi[e], err);
          lo[e] += err;
        }
      }
    } else if (live) {
      if constexpr (OUT == TIME_S) {
        float* dst = a.S + (size_t)p * F * a.out_nq + (a.out_qsel ? a.out_qsel[j] : j);
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int m = t + T * e;
          if (!BLUE || m < F) dst[(size_t)m * a.out_nq] = v[e].x * v[e].x + v[e].y * v[e].y;
        }
      } else {
        float2* dst = a.tilde + (size_t)p * F * a.nsel + j;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int m = t + T * e;
          if (!BLUE) dst[(size_t)m * a.nsel] = v[e];
          else if (m < F) dst[(size_t)m * a.nsel] = cmul(v[e], __ldg(a.chirp + m));
        }
      }
    }
    if (TC::PREFETCH) {
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = next[e];
      x0 = next0;
    } else if (!TC::ASYNC && tile + 1 < tile1) {
      load(v, x0, tile + 1);
    }
  }
  if constexpr (OUT == TIME_DETECTOR) {
    // over the columns, still as pairs and in an order fixed per bin
    int e0 = 0;
    bool writer = true;
    column_pairs<E, C / 2>(hi, lo, c, e0, writer);
    if (writer) {
#pragma unroll
      for (int e = 0; e < kept_bins(E, C); ++e) {
        const int m = t + T * (e0 + e);
        if (m < F)  // a sum past the largest float stays infinite
          a.part[((size_t)p * gridDim.x + blockIdx.x) * F + m] = (double)hi[e] + (isinf(hi[e]) ? 0.0 : (double)lo[e]);
      }
    }
  }
}

// Lengths with a kernel.
constexpr int kTimeLengths[] = {32, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1152, 2048, 4096};

int time_fft_length(int64_t F, bool* chirp) {
  for (int n : kTimeLengths)
    if (n == F && n <= 2048) {
      *chirp = false;
      return n;
    }
  *chirp = true;
  for (int n : kTimeLengths)
    if (fft_pow2(n) && n >= 2 * F - 1) return n;
  return 0;
}

namespace {

template <int N, int OUT, bool BLUE>
cudaError_t launch_n(TimeArgs a, cudaStream_t st) {
  using TC = TimeCfg<N, OUT, BLUE>;
  const int64_t tiles = (a.nsel + TC::C - 1) / TC::C;
  a.tpc = OUT == TIME_DETECTOR ? TIME_DET_TILES
                               : (int)std::min<int64_t>(8, std::max<int64_t>(1, tiles * a.P / (8 * 152 * TC::MINB)));
  const int64_t gx = (tiles + a.tpc - 1) / a.tpc;
  const int64_t gy = std::min<int64_t>(a.P, 65535), gz = (a.P + gy - 1) / gy;
  if (gx > 0x7fffffff || gz > 65535) return cudaErrorInvalidValue;
  auto* k = k_time_fft<N, OUT, BLUE>;
  if (TC::SMEM > 46 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, TC::SMEM);
    if (e != cudaSuccess) return e;
  }
  return launch_after(k, dim3((unsigned)gx, (unsigned)gy, (unsigned)gz), TC::THREADS, TC::SMEM, st, a);
}

template <int N>
cudaError_t launch_len(const TimeArgs& a, int out, bool chirp, cudaStream_t st) {
  if constexpr (fft_pow2(N)) {
    if (chirp) {
      if (out == TIME_S) return launch_n<N, TIME_S, true>(a, st);
      if (out == TIME_DETECTOR) return launch_n<N, TIME_DETECTOR, true>(a, st);
      return launch_n<N, TIME_TILDE, true>(a, st);
    }
  }
  if constexpr (N <= 2048) {
    if (out == TIME_S) return launch_n<N, TIME_S, false>(a, st);
    if (out == TIME_DETECTOR) return launch_n<N, TIME_DETECTOR, false>(a, st);
    return launch_n<N, TIME_TILDE, false>(a, st);
  }
  return cudaErrorInvalidValue;
}

#define TACAW_TIME_DISPATCH(n, CALL) \
  switch (n) {                       \
    case 32: return CALL(32);        \
    case 64: return CALL(64);        \
    case 96: return CALL(96);        \
    case 128: return CALL(128);      \
    case 192: return CALL(192);      \
    case 256: return CALL(256);      \
    case 384: return CALL(384);      \
    case 512: return CALL(512);      \
    case 768: return CALL(768);      \
    case 1024: return CALL(1024);    \
    case 1152: return CALL(1152);    \
    case 2048: return CALL(2048);    \
    case 4096: return CALL(4096);    \
  }

cudaError_t launch_time_fft(int n, const TimeArgs& a, int out, bool chirp, cudaStream_t st) {
#define TACAW_CALL(N) launch_len<N>(a, out, chirp, st)
  TACAW_TIME_DISPATCH(n, TACAW_CALL)
#undef TACAW_CALL
  return cudaErrorInvalidValue;
}

int64_t time_det_blocks(int n, bool chirp, int64_t nsel) {
  const int c = time_shape(n, TIME_DETECTOR, chirp).c * TIME_DET_TILES;
  return (nsel + c - 1) / c;
}

}  // namespace

int64_t time_fft_parts(int64_t F, int64_t nsel) {
  bool chirp;
  const int n = time_fft_length(F, &chirp);
  return n ? time_det_blocks(n, chirp, nsel) : 0;
}

// S (full, or the spectrum image with REDUCE_DETECTOR) by FFT; the caller has checked
// time_fft_length.
int spectrum_fft(tacaw_ctx* ctx, const float2* psi, int64_t P, int64_t F, const SpecIO& io, int32_t reduce, float* S,
                 Scratch& sc) {
  TimeArgs a{};
  bool chirp;
  const int n = time_fft_length(F, &chirp);
  a.psi = psi;
  a.P = P;
  a.F = a.nf = F;
  a.in_nq = io.in_nq;
  a.in_qsel = io.in_qsel;
  a.nsel = io.nsel;
  a.out_nq = io.out_nq;
  a.out_qsel = io.out_qsel;
  a.tw = ctx->tw;
  a.S = S;
  if (chirp) {
    const int rc = get_chirp(ctx, F, n, &a.chirp, &a.bhat);
    if (rc != TACAW_OK) return rc;
  }
  const bool det = reduce == TACAW_REDUCE_DETECTOR;
  const int64_t nparts = det ? time_det_blocks(n, chirp, io.nsel) : 0;
  cudaError_t e;
  if (det && (e = sc.get(&a.part, (size_t)P * nparts * F)) != cudaSuccess)
    return cuda_err(ctx, e, "detector partial sums");
  const double pfq = (double)P * F * io.nsel;
  {
    ProfScope ps(ctx, "time_fft", sc.st, pfq * 8 + (det ? (double)P * nparts * F * 8 : pfq * 4),
                 pfq * 5.0 * std::log2((double)std::max<int64_t>(F, 2)));
    if ((e = launch_time_fft(n, a, det ? TIME_DETECTOR : TIME_S, chirp, sc.st)) != cudaSuccess)
      return cuda_err(ctx, e, "k_time_fft");
  }
  if (det) {
    ProfScope ps(ctx, "detector_tiles", sc.st, (double)P * nparts * F * 8 + (double)P * F * 4, (double)P * nparts * F);
    if ((e = launch_detector_parts(a.part, P, F, nparts, S, sc.st)) != cudaSuccess)
      return cuda_err(ctx, e, "k_detector_parts");
  }
  return TACAW_OK;
}

// psi~ of the frames [f0, f0 + nf) of F against a static reference (tacaw_spectrum_partial).
int partial_fft(tacaw_ctx* ctx, const float2* psi, const float2* ref, int64_t P, int64_t nf, int64_t f0, int64_t F,
                int64_t nq, const int32_t* qsel, int64_t nsel, float2* tilde, cudaStream_t st) {
  TimeArgs a{};
  bool chirp;
  const int n = time_fft_length(F, &chirp);
  a.psi = psi;
  a.ref = ref;
  a.P = P;
  a.F = F;
  a.nf = nf;
  a.f0 = f0;
  a.in_nq = nq;
  a.in_qsel = qsel;
  a.nsel = nsel;
  a.tilde = tilde;
  a.tw = ctx->tw;
  if (chirp) {
    const int rc = get_chirp(ctx, F, n, &a.chirp, &a.bhat);
    if (rc != TACAW_OK) return rc;
  }
  ProfScope ps(ctx, "time_fft_partial", st, (double)P * nsel * 8 * (nf + F),
               (double)P * nsel * F * 5.0 * std::log2((double)std::max<int64_t>(F, 2)));
  const cudaError_t e = launch_time_fft(n, a, TIME_TILDE, chirp, st);
  return e == cudaSuccess ? TACAW_OK : cuda_err(ctx, e, "k_time_fft");
}

}  // namespace tacaw
