// Slice kernels: binning, projected potential, transmission, probe and the multislice step.
//
// Every 2D transform is a row pass (FFT along x inside one CTA per G rows) followed by a column
// pass (FFT along y inside one CTA per C columns); pointwise work is fused into the passes:
//   potential  (Methods, "Atomic Scattering Potentials"):
//     spread atoms -> FFT_x | FFT_y, * C M (f_A - i f_B)/Phi, IFFT_y | IFFT_x, Re -> V
//   transmission (Methods, "Multislice Propagation", t = exp(i sigma V)):
//     exp(i sigma V) -> FFT_x | FFT_y, * M / Nq, IFFT_y | IFFT_x -> t
//   slice step  (same section, psi <- IDFT(P M DFT(t psi))):
//     [IFFT_x] * t, FFT_x | FFT_y, * P M / Nq, IFFT_y    (the IFFT_x of slice s is fused into
//     the row pass of slice s+1; the last column pass writes psi(k) without the inverse)
// Between the passes only the in-band columns (|kx| <= kbl) are kept, in compact order.
#include <cuda_runtime.h>

#include <algorithm>

#include "fft.cuh"
#include "tacaw_internal.cuh"

namespace tacaw {

// Per-kernel variants of the FFT pass kernels, chosen per transform length by the autotuner
// (paper_2602_10064_gb300/tune.py), which times every variant on GB300 and writes
// tuning_table.h.  Variant bits: 2 = 1.5 to 2 times as many resident threads per SM (fewer
// registers each), 4 = column passes only: twice the columns per CTA, so that each load
// instruction covers whole 128-byte lines, 8 = 32 elements per thread for the powers of two from
// 128 points (two-pass transforms, about 170 registers).  TACAW_TUNE_FORCE=v builds every kernel
// as variant v (the tuner's measurement builds).
enum KernelId {
  K_SPLAT_ROW, K_COL_POT, K_ROW_POT_OUT, K_ROW_VT, K_COL_T, K_ROW_TOUT, K_PROBE_COL, K_PROBE_ROW,
  K_SLICE_ROW, K_SLICE_COL, K_SLICE_ROW_SCAN
};
}  // namespace tacaw
#include "tuning_table.h"
namespace tacaw {
#ifndef TACAW_TUNE_FORCE
#define TACAW_TUNE_FORCE -1
#endif
template <int K, int N>
struct Tuned {
  static constexpr int V = TACAW_TUNE_FORCE >= 0 ? TACAW_TUNE_FORCE : tuned_variant(K, N);
  static constexpr bool COLUMN = K == K_COL_POT || K == K_COL_T || K == K_PROBE_COL || K == K_SLICE_COL;
  static constexpr int EV = (V & 8) ? 1 : 0;
  static constexpr int WIDE = (COLUMN && (V & 4)) ? 1 : 0;
  // resident CTAs per SM requested for a CTA of `threads`: `target` threads per SM; variant & 2: 1.5
  // times as many, or twice where that makes no difference to the CTAs and in the spreading pass
  __host__ __device__ static constexpr int minb(int threads, int target) {
    const int base = target / threads, more = target * 3 / 2 / threads, most = target * 2 / threads;
    const int n = !(V & 2) ? base : K == K_SPLAT_ROW || more == base ? most : more;
    return n > 1 ? n : 1;
  }
};

// Largest power of two <= x (x >= 1).
__host__ __device__ constexpr int floor_pow2(int x) {
  int p = 1;
  while (2 * p <= x) p *= 2;
  return p;
}

// Row passes: G rows per CTA, one transform group of T threads per row.  Transforms of 24
// elements per thread need about 170 registers, so those CTAs are smaller and the SM holds
// 384 instead of 512 threads (TARGET).
// EV = 1: 32 elements per thread (two-pass transforms) for the powers of two from 128 points.
// SMALL and LARGE, threads per CTA with up to 16 elements each and with more: the spreading pass takes 256
// and 192, to share its candidate tables over more rows, the others 64 and 192: small CTAs keep the phases
// of an SM's warps apart.  256-point slice row pass of a probe scan, 160 launches: 48.3 ms with 256
// threads, 45.7 with 128, 44.3 with 64.  The slice row pass takes 96 where a row lies in half a warp (512
// points 4.01 ps a point with 192, 3.76 with 96; 384 points 4.53, 4.40); not above that, where it has to
// synchronise several warps (768 points 4.33, 4.43; 1152 points 4.81, 4.90).
template <int N, int EV = 0, int SMALL = 64, int LARGE = 192>
struct RowCfg {
  static constexpr int E = (EV && fft_pow2(N) && N >= 128) ? 32 : FftPlan<N>::E;
  static constexpr int T = N / E;
  static constexpr int TARGET = E >= 24 ? 384 : 512;
  static constexpr int G0 = (E < 24 ? SMALL : T < 32 ? LARGE : 192) / T;
  static constexpr int G = G0 > 32 ? 32 : (G0 < 1 ? 1 : floor_pow2(G0));  // rows per CTA
  static constexpr int THREADS = G * T;
  static constexpr int SMEM = G * row_smem_stride<N, E>() * (int)sizeof(float2);
};

// Column passes: C columns per CTA (WIDE doubles C).  With 8 or 16 elements a thread, 128 threads but
// at least 16 columns (whole 128-byte lines) where 256 threads hold them: 64 points 5.85 -> 4.94 and
// 128 points 3.23 -> 2.97 ps a point in the slice pass; 256 points lose 5% with 8 columns.
template <int N, int WIDE = 0, int EV = 0>
struct ColCfg {
  static constexpr int E = (EV && fft_pow2(N) && N >= 128) ? 32 : FftPlan<N>::E;
  static constexpr int T = N / E;
  static constexpr int TARGET = E >= 24 ? 384 : 512;
  static constexpr int FULL = TARGET / 2 / T, HALF = TARGET / 4 / T;
  static constexpr int C0 = (E >= 24 || FULL <= 16 ? FULL : HALF < 16 ? 16 : HALF) << WIDE;
  static constexpr int C = C0 > 32 ? 32 : (C0 < 4 ? 4 : floor_pow2(C0));  // columns per CTA (divides Wp)
  static constexpr int THREADS = C * T;
  // padding of the interleaved columns: pays only with 32 elements per thread (with 8 columns of 1152
  // points it saves 20% of the exchanges' wavefronts, but the pass takes 264 us instead of 218)
  static constexpr int SH = E == 32 ? 5 : 0;
  static constexpr int SMEM = (N + (SH ? (N >> SH) : 0)) * C * (int)sizeof(float2);
};

// The configuration of each pass kernel; a kernel and its launcher name the same alias.
template <int N> using SplatCfg = RowCfg<N, Tuned<K_SPLAT_ROW, N>::EV, 256>;
template <int N> using PotOutCfg = RowCfg<N, Tuned<K_ROW_POT_OUT, N>::EV>;
template <int N> using RowVtCfg = RowCfg<N, Tuned<K_ROW_VT, N>::EV>;
template <int N> using RowToutCfg = RowCfg<N, Tuned<K_ROW_TOUT, N>::EV>;
template <int N> using ProbeRowCfg = RowCfg<N, Tuned<K_PROBE_ROW, N>::EV>;
// one probe (the compact t, TF) and several (the full t) have different loops: tuned apart
template <bool TF> __host__ __device__ constexpr int slice_row_id() { return TF ? K_SLICE_ROW : K_SLICE_ROW_SCAN; }
template <int N, bool TF> using SliceRowCfg = RowCfg<N, Tuned<slice_row_id<TF>(), N>::EV, 64, 96>;
template <int N> using ColPotCfg = ColCfg<N, Tuned<K_COL_POT, N>::WIDE, Tuned<K_COL_POT, N>::EV>;
template <int N> using ColTCfg = ColCfg<N, Tuned<K_COL_T, N>::WIDE, Tuned<K_COL_T, N>::EV>;
template <int N> using ProbeColCfg = ColCfg<N, Tuned<K_PROBE_COL, N>::WIDE, Tuned<K_PROBE_COL, N>::EV>;
template <int N> using SliceColCfg = ColCfg<N, Tuned<K_SLICE_COL, N>::WIDE, Tuned<K_SLICE_COL, N>::EV>;

// Resident CTAs per SM requested from the compiler for kernel K with configuration Cfg.
template <int K, int N, class Cfg>
__host__ __device__ constexpr int minb_of() {
  return Tuned<K, N>::minb(Cfg::THREADS, Cfg::TARGET);
}

// Barrier of one row transform: the group's own (warp, or named barrier over whole warps), or one of
// the two groups that fill whole warps together (T = 48: 1152 points).
template <int T>
__device__ __forceinline__ auto group_sync(int g) {
  if constexpr (T <= 32 || T % 32 == 0) return GroupSync<T>{1 + g};
  else return GroupSync<2 * T>{1 + g / 2};
}

// CTAs of a column pass: the in-band columns c < W only, C per CTA.  The padding columns up to Wp
// are never read by a row pass (no x maps to them), so they need no transform.
static int col_blocks(const Band& b, int C) { return (b.W + C - 1) / C; }

// Batch index over (grid.y, grid.z); batches beyond nb return before any barrier.
__device__ __forceinline__ int batch_index() { return blockIdx.y + gridDim.y * blockIdx.z; }
static dim3 batch_grid(int gx, int64_t nb) {
  unsigned y = (unsigned)(nb < 65535 ? nb : 65535);
  unsigned z = (unsigned)((nb + y - 1) / y);
  return dim3((unsigned)gx, y, z);
}

// The compact row accessors with the band read at run time.  Elements e < E / 2 cover x < N / 2,
// where only x <= mb is in band (c = x), the others x >= N / 2, where only x >= N - mb is
// (c = x - N + W; with every column kept, mb = N / 2 and W = N, c = x): one comparison of t with a
// value common to all threads, and a fixed offset from one of two pointers.
template <int N, int E>
__device__ __forceinline__ void load_row_compact(float2 (&v)[E], const float2* __restrict__ src, const Band& b,
                                                 int t) {
  constexpr int T = N / E;
  const float2 *lo = src + t, *hi = src + t + (b.W - N);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const bool in = e < E / 2 ? t <= b.mb - T * e : t >= N - b.mb - T * e;
    v[e] = in ? (e < E / 2 ? lo : hi)[T * e] : make_float2(0.f, 0.f);
  }
}

template <int N, int E>
__device__ __forceinline__ void store_row_compact(const float2 (&v)[E], float2* __restrict__ dst, const Band& b,
                                                  int t) {
  constexpr int T = N / E;
  float2 *lo = dst + t, *hi = dst + t + (b.W - N);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const bool in = e < E / 2 ? t <= b.mb - T * e : t >= N - b.mb - T * e;
    if (in) (e < E / 2 ? lo : hi)[T * e] = v[e];
  }
}

// The same with the band's half-width MB known at compile time (W = 2 MB + 1): the element e of
// every thread covers positions [T e, T e + T), so whether it is in band, out of band or split
// is decided per e at compile time, and only the split elements keep a per-thread test.
template <int N, int E, int MB>
__device__ __forceinline__ void load_row_band(float2 (&v)[E], const float2* __restrict__ src, int t) {
  constexpr int T = N / E, W = 2 * MB + 1;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int x = t + T * e;
    if (T * e + T - 1 <= MB) {
      v[e] = src[x];
    } else if (T * e >= N - MB) {
      v[e] = src[x - N + W];
    } else if (T * e > MB && T * e + T - 1 < N - MB) {
      v[e] = make_float2(0.f, 0.f);
    } else {
      const int c = x <= MB ? x : (x >= N - MB ? x - N + W : -1);
      v[e] = c >= 0 ? src[c] : make_float2(0.f, 0.f);
    }
  }
}

template <int N, int E, int MB>
__device__ __forceinline__ void store_row_band(const float2 (&v)[E], float2* __restrict__ dst, int t) {
  constexpr int T = N / E, W = 2 * MB + 1;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int x = t + T * e;
    if (T * e + T - 1 <= MB) {
      dst[x] = v[e];
    } else if (T * e >= N - MB) {
      dst[x - N + W] = v[e];
    } else if (!(T * e > MB && T * e + T - 1 < N - MB)) {
      const int c = x <= MB ? x : (x >= N - MB ? x - N + W : -1);
      if (c >= 0) dst[c] = v[e];
    }
  }
}

// The compact row accessors with the band's half-width fixed at compile time (MB >= 0) or
// read from b (MB < 0).
template <int N, int MB, int E>
__device__ __forceinline__ void load_row(float2 (&v)[E], const float2* __restrict__ src, const Band& b, int t) {
  if constexpr (MB >= 0) load_row_band<N, E, MB>(v, src, t);
  else load_row_compact<N>(v, src, b, t);
}
template <int N, int MB, int E>
__device__ __forceinline__ void store_row(const float2 (&v)[E], float2* __restrict__ dst, const Band& b, int t) {
  if constexpr (MB >= 0) store_row_band<N, E, MB>(v, dst, t);
  else store_row_compact<N>(v, dst, b, t);
}

// ============================================================================================
// a1: slice binning.  Slice, grid cell and offset of every atom, then one CTA per frame scatters
// stably, so every slice list keeps atom order.
// ============================================================================================
constexpr int BIN_THREADS = 1024;
constexpr int BIN_MAX_S = 256;

// x wrapped into [0, L): x - L floor(x / L), every operation rounded.  Within one cell length of the
// cell the rounded quotient lies strictly between the same integers as the exact one, so its floor
// is known from comparisons; the FP64 division is left to positions farther out.
__device__ __forceinline__ double wrap_cell(double x, double L) {
  if (x >= 0.0 && x < L) return x;
  if (x >= -L && x < 0.0) return __dsub_rn(x, -L);
  if (x >= L && x < 2.0 * L) return __dsub_rn(x, L);
  return __dsub_rn(x, __dmul_rn(L, floor(x / L)));
}

// floor(z_w / dz): from the product with 1 / dz (off by less than 1e-12 for S <= 256) where that is
// clear of an integer, else from the division.
__device__ __forceinline__ int slice_of(double z, const BinGeom& g) {
  const double zw = wrap_cell(z, g.Lz), q = __dmul_rn(zw, g.inv_dz), fq = floor(q), fr = __dsub_rn(q, fq);
  int s = fr > 1e-9 && fr < 1.0 - 1e-9 ? (int)fq : (int)floor(zw / g.dz);
  if (s >= g.S) s = g.S - 1;
  if (s < 0) s = 0;
  return s;
}

// The index stays in [0, n) for every x: 0 where x is not finite (its fraction is NaN, which the spreading
// kernel takes as out of reach: the atom adds nothing) or too far out for FP64 to wrap.
__device__ __forceinline__ void grid_coord(double x, double L, double per_len, int n, int& i0, float& fr) {
  const double u = __dmul_rn(wrap_cell(x, L), per_len);
  double fl = floor(u);
  int i = (int)fl;
  double f = __dsub_rn(u, fl);
  if (i >= n) { i -= n; }
  if (i < 0) { i += n; }
  i0 = i >= 0 && i < n ? i : 0;
  fr = (float)f;
}

// Slice of every atom (tacaw_bin_slices).
__global__ void __launch_bounds__(256) k_slice_index(const float* __restrict__ pos, int64_t n, BinGeom g,
                                                     int* __restrict__ slice_out) {
  const int64_t j = blockIdx.x * (int64_t)256 + threadIdx.x;
  if (j < n) slice_out[j] = slice_of((double)pos[3 * j + 2], g);
}

// Record and slice of every atom, in atom order, one thread each: the FP64 work of the binning
// (GB300 issues two FP64 operations a clock and SM) spread over the whole chip.  With it inside the
// one CTA per frame that scatters, and with seven divisions an atom, 12 frames of 8000 atoms took
// 190 us; this and the scatter take 33.
__global__ void __launch_bounds__(256) k_atoms(const float* __restrict__ pos, int A, int64_t nf, BinGeom g,
                                               const int8_t* __restrict__ slot_of_atom, AtomRec* __restrict__ rec,
                                               uint8_t* __restrict__ key) {
  grid_dependency_wait();
  const int j = blockIdx.x * 256 + threadIdx.x;
  if (j >= A || batch_index() >= nf) return;
  const size_t at = (size_t)batch_index() * A + j;
  const float* P = pos + 3 * at;
  AtomRec r;
  int ix, iy;
  grid_coord((double)P[0], g.Lx, g.per_x, g.nx, ix, r.fx);
  grid_coord((double)P[1], g.Ly, g.per_y, g.ny, iy, r.fy);
  r.ixy = ix | (iy << 16);
  r.jslot = j | ((int)slot_of_atom[j] << 24);
  rec[at] = r;
  key[at] = (uint8_t)slice_of((double)P[2], g);
}

__global__ void __launch_bounds__(BIN_THREADS) k_bin(const AtomRec* __restrict__ rec, const uint8_t* __restrict__ key,
                                                      int A, int S, AtomRec* __restrict__ recs,
                                                      int* __restrict__ offs) {
  grid_dependency_wait();
  __shared__ int counts[BIN_MAX_S];
  __shared__ int cursor[BIN_MAX_S];
  __shared__ int wcount[BIN_THREADS / 32][BIN_MAX_S];
  const int f = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint8_t* K = key + (size_t)f * A;
  for (int s = tid; s < S; s += BIN_THREADS) counts[s] = 0;
  __syncthreads();
  for (int j = tid; j < A; j += BIN_THREADS) atomicAdd(&counts[K[j]], 1);
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int s = 0; s < S; ++s) {
      offs[(size_t)f * (S + 1) + s] = run;
      cursor[s] = run;
      run += counts[s];
    }
    offs[(size_t)f * (S + 1) + S] = run;
  }
  const unsigned lt = (1u << lane) - 1u;
  for (int base = 0; base < A; base += BIN_THREADS) {
    for (int i = tid; i < (BIN_THREADS / 32) * S; i += BIN_THREADS) wcount[i / S][i % S] = 0;
    __syncthreads();
    const int j = base + tid;
    const bool valid = j < A;
    const int s = valid ? K[j] : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, s);
    const int rank = __popc(peers & lt);
    if (valid && rank == 0) wcount[w][s] = __popc(peers);
    __syncthreads();
    for (int ss = tid; ss < S; ss += BIN_THREADS) {
      int run = cursor[ss];
      for (int ww = 0; ww < BIN_THREADS / 32; ++ww) {
        const int c = wcount[ww][ss];
        wcount[ww][ss] = run;
        run += c;
      }
      cursor[ss] = run;
    }
    __syncthreads();
    if (valid) recs[(size_t)f * A + wcount[w][s] + rank] = rec[(size_t)f * A + j];
    __syncthreads();
  }
}

__global__ void k_map_slots(const int32_t* __restrict__ Z, int64_t A, const int8_t* __restrict__ lut,
                            int8_t* __restrict__ slot, int* __restrict__ status) {
  grid_dependency_wait();
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < A; j += (int64_t)gridDim.x * blockDim.x) {
    const int z = Z[j];
    int s = (z >= 0 && z < 256) ? lut[z] : -1;
    if (s < 0) {
      atomicOr(status, TACAW_STATUS_SPECIES);
      s = 0;
    }
    slot[j] = (int8_t)s;
  }
}

cudaError_t launch_map_slots(const int32_t* Z, int64_t A, const int8_t* lut, int8_t* slot, int* status,
                             cudaStream_t st) {
  if (A <= 0) return cudaSuccess;
  const int64_t blocks = (A + 255) / 256;
  return launch_after(k_map_slots, (unsigned)(blocks < 1024 ? blocks : 1024), 256, 0, st, Z, A, lut, slot, status);
}

// One warp per (frame, slice): stable counting sort of the slice's atom records by the grid
// row of their coordinate, and the offsets of each block of SPREAD_YB rows, so that the
// spreading pass reads only the atoms whose footprint can reach its rows.  Order within a row
// is the binning order (atom index), so the spreading sums stay deterministic.
constexpr int SORT_WARPS = 8;
__global__ void __launch_bounds__(SORT_WARPS * 32)
    k_sort_rows(const AtomRec* __restrict__ recs, const int* __restrict__ offs, int A, int S, int nseg, int ny,
                AtomRec* __restrict__ out, int* __restrict__ boffs) {
  grid_dependency_wait();
  extern __shared__ int cnt_all[];  // [SORT_WARPS][ny]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int seg = blockIdx.x * SORT_WARPS + warp;
  if (seg >= nseg) return;  // whole warps; only warp-level barriers below
  int* cnt = cnt_all + warp * ny;
  const int f = seg / S, s = seg - f * S;
  const int lo = offs[(size_t)f * (S + 1) + s], hi = offs[(size_t)f * (S + 1) + s + 1];
  const AtomRec* R = recs + (size_t)f * A;
  AtomRec* O = out + (size_t)f * A;
  const int nyb = ny / SPREAD_YB;
  int* bo = boffs + (size_t)seg * (nyb + 1);
  for (int y = lane; y < ny; y += 32) cnt[y] = 0;
  __syncwarp();
  for (int j = lo + lane; j < hi; j += 32) atomicAdd(&cnt[R[j].ixy >> 16], 1);
  __syncwarp();
  int run = lo;  // exclusive scan over rows; block offsets at multiples of SPREAD_YB
  for (int y0 = 0; y0 < ny; y0 += 32) {
    const int y = y0 + lane;
    const int c = y < ny ? cnt[y] : 0;
    int x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += n;
    }
    if (y < ny) {
      cnt[y] = run + x - c;
      if (y % SPREAD_YB == 0) bo[y / SPREAD_YB] = run + x - c;
    }
    run += __shfl_sync(0xffffffffu, x, 31);
  }
  if (lane == 0) bo[nyb] = hi;
  __syncwarp();
  const unsigned below = (1u << lane) - 1u;
  for (int base = lo; base < hi; base += 32) {  // 32 records at a time, in order: stable
    const int j = base + lane;
    const bool valid = j < hi;
    AtomRec r;
    int key = -1 - lane;  // distinct for the lanes past the end
    if (valid) {
      r = R[j];
      key = r.ixy >> 16;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    const int leader = __ffs(peers) - 1;
    int pos = 0;
    if (valid && lane == leader) {
      pos = cnt[key];
      cnt[key] = pos + __popc(peers);
    }
    pos = __shfl_sync(0xffffffffu, pos, leader) + __popc(peers & below);
    if (valid) O[pos] = r;
    __syncwarp();
  }
}

cudaError_t launch_sort_rows(const AtomRec* recs, const int* offs, int64_t A, int64_t nf, int S, int ny,
                             AtomRec* out, int* boffs, cudaStream_t st) {
  if (ny % SPREAD_YB != 0 || nf <= 0) return cudaErrorInvalidValue;
  const int64_t nseg = nf * S;
  const int smem = SORT_WARPS * ny * (int)sizeof(int);
  if (smem > 46 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_sort_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  return launch_after(k_sort_rows, (unsigned)((nseg + SORT_WARPS - 1) / SORT_WARPS), SORT_WARPS * 32, smem, st, recs,
                      offs, (int)A, S, (int)nseg, ny, out, boffs);
}

cudaError_t launch_slice_index(const float* pos, int64_t n, const BinGeom& g, int* slice_out, cudaStream_t st) {
  if (g.S > BIN_MAX_S || n <= 0 || (n + 255) / 256 > 0x7fffffff) return cudaErrorInvalidValue;
  k_slice_index<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(pos, n, g, slice_out);
  return cudaGetLastError();
}

cudaError_t launch_bin(const float* pos, int64_t A, int64_t nf, const BinGeom& g, const int8_t* slot_of_atom,
                       AtomRec* rec, uint8_t* key, AtomRec* recs, int* offs, cudaStream_t st) {
  if (g.S > BIN_MAX_S || nf <= 0) return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
  if (A > 0)
    e = launch_after(k_atoms, batch_grid((int)((A + 255) / 256), nf), 256, 0, st, pos, (int)A, nf, g, slot_of_atom, rec,
                     key);
  if (e != cudaSuccess) return e;
  return launch_after(k_bin, (unsigned)nf, BIN_THREADS, 0, st, rec, key, (int)A, g.S, recs, offs);
}

// ============================================================================================
// a2: potential.  Row pass: spread the atoms of one slice and one species pair onto G rows
// (gather per grid point, candidates in atom order, so the sum is deterministic), then FFT_x.
// ============================================================================================
// x mod n for 0 <= x < 3 n (any n, no division).
__device__ __forceinline__ int wrap3(int x, int n) {
  x -= (x >= n) ? n : 0;
  return x - ((x >= n) ? n : 0);
}
// The same for a compile-time n (a mask when n is a power of two).
template <int N>
__device__ __forceinline__ int wrap3(int x) {
  if constexpr (fft_pow2(N)) return x & (N - 1);
  else return wrap3(x, N);
}

__device__ __forceinline__ float es_kernel(float z, float beta) {
  const float a = 1.f - z * z;
  return a > 0.f ? expf(beta * (sqrtf(a) - 1.f)) : 0.f;
}

// Shared memory of the spreading row pass: per-row accumulators (each element owned by one
// thread, so the sums are race-free and in candidate order), then the candidate tables.
template <int NX>
struct SplatSmem {
  static constexpr int NT = SplatCfg<NX>::THREADS, G = SplatCfg<NX>::G;
  static constexpr int ACC = G * NX * 8;
  static constexpr int TAB = NT * (2 * SPREAD_HALF + G) * 4 + NT * 5 * 4;
  static constexpr int BYTES = (ACC + TAB) > SplatCfg<NX>::SMEM ? (ACC + TAB) : SplatCfg<NX>::SMEM;
};

template <int NX, int MB = -1>
__global__ void __launch_bounds__(SplatCfg<NX>::THREADS, minb_of<K_SPLAT_ROW, NX, SplatCfg<NX>>())
    k_splat_row(Geo geo, Band b, const AtomRec* __restrict__ recs, const int* __restrict__ boffs, int A, int S,
                int s0, int sb, int npair, int two, int nbatch, float beta, float2* __restrict__ Bp) {
  grid_dependency_wait();
  constexpr int E = SplatCfg<NX>::E, T = SplatCfg<NX>::T, G = SplatCfg<NX>::G, NT = SplatCfg<NX>::THREADS;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);                     // FFT scratch (after spreading)
  float2* acc = reinterpret_cast<float2*>(smraw);                    // [G][NX]
  constexpr int h = SPREAD_HALF, W2 = 2 * h;
  float* phx = reinterpret_cast<float*>(smraw + SplatSmem<NX>::ACC); // [NT][W2]
  float* phy = phx + NT * W2;                                         // [NT][G]
  float* cfx = phy + NT * G;                                          // [NT] candidate records
  float* cfy = cfx + NT;
  int* cx0 = reinterpret_cast<int*>(cfy + NT);                        // first footprint column, | imag << 16
  int* ciy = cx0 + NT;                                                // iy0, -1: other pair
  int* crow = ciy + NT;                                               // iy0 - y0, unwrapped

  const int bidx = batch_index();
  if (bidx >= nbatch) return;
  // two: the planes are pairs of slices (2i, 2i + 1) of the one species, the second as imaginary part;
  // else slices, the odd slots of a species pair as imaginary part
  const int pair = bidx % npair, fs = bidx / npair, f = fs / sb;
  const int sa = two ? 2 * (s0 / 2 + fs % sb) : s0 + fs % sb, nhalf = two && sa + 1 < S ? 2 : 1;
  const int tid = threadIdx.x, g = tid / T, t = tid % T;
  const int ny = geo.ny, y0 = blockIdx.x * G;
  const AtomRec* R = recs + (size_t)f * A;
  // candidates: the atoms of the row blocks covering rows [y0 - h, y0 + G - 2 + h] (their
  // footprints [iy0 + 1 - h, iy0 + h] meet rows [y0, y0 + G)), at most two contiguous ranges of
  // the row-sorted slice list (the window may wrap around y = 0)
  const int nyb = ny / SPREAD_YB;
  const int wlo = y0 - h, whi = y0 + G - 2 + h;
  const int b_lo = wlo >= 0 ? wlo / SPREAD_YB : -((-wlo + SPREAD_YB - 1) / SPREAD_YB), b_hi = whi / SPREAD_YB;
  const bool whole = b_hi - b_lo + 1 >= nyb;

#pragma unroll
  for (int e = 0; e < E; ++e) acc[g * NX + t + T * e] = make_float2(0.f, 0.f);

  for (int half = 0; half < nhalf; ++half) {
    const int* bo = boffs + ((size_t)f * S + sa + half) * (nyb + 1);
    int s1, n1, s2 = 0, n2 = 0;
    if (whole) {
      s1 = bo[0];
      n1 = bo[nyb] - s1;
    } else if (b_lo < 0) {
      s1 = bo[b_lo + nyb];
      n1 = bo[nyb] - s1;
      s2 = bo[0];
      n2 = bo[b_hi + 1] - s2;
    } else if (b_hi >= nyb) {
      s1 = bo[b_lo];
      n1 = bo[nyb] - s1;
      s2 = bo[0];
      n2 = bo[b_hi - nyb + 1] - s2;
    } else {
      s1 = bo[b_lo];
      n1 = bo[b_hi + 1] - s1;
    }
    const int M = n1 + n2;

    for (int base = 0; base < M; base += NT) {
      // 1. the batch's candidate records (atoms of other species pairs are marked and skipped)
      const int j = base + tid;
      if (j < M) {
        const AtomRec r = R[j < n1 ? s1 + j : s2 + (j - n1)];
        const int slot = r.jslot >> 24;
        cfx[tid] = r.fx;
        cfy[tid] = r.fy;
        cx0[tid] = wrap3<NX>((r.ixy & 0xffff) + 1 - h + NX) | ((two ? half : slot & 1) << 16);
        const int iy = r.ixy >> 16;
        ciy[tid] = (slot >> 1) == pair ? iy : -1;
        int dy = iy - SPREAD_YB * b_lo;  // rows above the first candidate block
        dy += dy < 0 ? ny : 0;
        crow[tid] = dy - (dy >= ny ? ny : 0) + SPREAD_YB * b_lo - y0;
      }
      __syncthreads();
      const int total = M - base < NT ? M - base : NT;
      // 2. kernel tables, one entry per thread: phx[c][d] (d < 2h) and phy[c][g]
      const int per = W2 + G;
      for (int i = tid; i < total * per; i += NT) {
        const int c = i / per, k = i - c * per;
        if (k < W2) {
          phx[c * W2 + k] = es_kernel(((float)(k + 1 - h) - cfx[c]) / (float)h, beta);
        } else {
          const int gg = k - W2, cy = ciy[c];
          int d = wrap3(y0 + gg - cy + ny, ny);
          if (d > ny / 2) d -= ny;
          phy[c * G + gg] = (cy >= 0 && d >= 1 - h && d <= h) ? es_kernel(((float)d - cfy[c]) / (float)h, beta)
                                                             : 0.f;
        }
      }
      __syncthreads();
      // 3. taps: thread (g, t) owns columns t + T e; a footprint of 2h columns starting at x0
      //    meets them at the offsets congruent to t - x0 modulo T.  The candidates come in row order
      //    (when they are not the whole slice), so those whose footprints hold this warp's rows are
      //    one run of them; walking all of them took 512 points x
      //    128 slices 117 us, this 99.
      int c0 = 0, c1 = total;
      if (!whole) {
        const int lane = tid & 31, g0 = (tid - lane) / T, g1 = (tid - lane + 31) / T;  // rows of this warp
        c1 = 0;
        for (int c = 0; c < total; c += 32) {
          const int r = c + lane < total ? crow[c + lane] : ny;
          c0 += __popc(__ballot_sync(0xffffffffu, r < g0 - h));
          c1 += __popc(__ballot_sync(0xffffffffu, r <= g1 - 1 + h));
        }
      }
      float* arow = reinterpret_cast<float*>(acc + g * NX);
      float wy = c0 < c1 ? phy[c0 * G + g] : 0.f;
      int xi = c0 < c1 ? cx0[c0] : 0;
      for (int c = c0; c < c1; ++c) {
        const float wyc = wy;
        const int x0 = xi & 0xffff, im = xi >> 16;
        if (c + 1 < c1) {
          wy = phy[(c + 1) * G + g];
          xi = cx0[c + 1];
        }
        if (wyc == 0.f) continue;
        const int d = wrap3<NX>(x0 - t + NX);
        for (int off = (T - d % T) % T; off < W2; off += T)
          arow[2 * wrap3<NX>(x0 + off) + im] += wyc * phx[c * W2 + off];
      }
      __syncthreads();
    }
  }
  float2 v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = acc[g * NX + t + T * e];
  __syncthreads();  // the FFT scratch of one group overlaps the accumulators of the next
  fft<NX, -1>(v, sm, RowIdx<NX, E>{g * row_smem_stride<NX, E>()}, t, geo.tw,
                  group_sync<T>(g));
  store_row<NX, MB>(v, Bp + ((size_t)bidx * ny + y0 + g) * b.Wp, b, t);
}

// Column pass of the potential: per (f, s), sum over species pairs of mtab * FFT_y, then IFFT_y.
template <int NY, bool ONE, int WPC = -1>
__global__ void __launch_bounds__(ColPotCfg<NY>::THREADS, minb_of<K_COL_POT, NY, ColPotCfg<NY>>())
    k_col_pot(Geo geo, Band b, const float2* __restrict__ Bp, const float2* __restrict__ mtab, int npair, int nbatch,
              float2* __restrict__ Ap) {
  grid_dependency_wait();
  using CC = ColPotCfg<NY>;
  constexpr int E = CC::E, T = CC::T, C = CC::C;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int fs = batch_index();
  if (fs >= nbatch) return;
  const int Wp = WPC > 0 ? WPC : b.Wp;
  const int c = threadIdx.x % C, t = threadIdx.x / C, cc = blockIdx.x * C + c;
  const ColIdx<C, CC::SH> idx{c};
  const BlockSync sync;
  const float2* tw = geo.tw;
  if constexpr (ONE) {
    // one species pair: no accumulator held across the transforms
    const float2* src = Bp + (size_t)fs * NY * Wp + cc;
    float2 v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = src[(size_t)(t + T * e) * Wp];
    fft<NY, -1>(v, sm, idx, t, tw, sync);
    const float2* m = mtab + cc;
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = cmul(m[(size_t)(t + T * e) * Wp], v[e]);
    fft<NY, +1>(v, sm, idx, t, tw, sync);
    float2* dst = Ap + (size_t)fs * NY * Wp + cc;
#pragma unroll
    for (int e = 0; e < E; ++e) dst[(size_t)(t + T * e) * Wp] = v[e];
  } else {
    float2 acc[E];
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = make_float2(0.f, 0.f);
    for (int pr = 0; pr < npair; ++pr) {
      const float2* src = Bp + (size_t)(fs * npair + pr) * NY * Wp + cc;
      float2 v[E];
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = src[(size_t)(t + T * e) * Wp];
      fft<NY, -1>(v, sm, idx, t, tw, sync);
      const float2* m = mtab + (size_t)pr * NY * Wp + cc;
#pragma unroll
      for (int e = 0; e < E; ++e) acc[e] = acc[e] + cmul(m[(size_t)(t + T * e) * Wp], v[e]);
    }
    fft<NY, +1>(acc, sm, idx, t, tw, sync);
    float2* dst = Ap + (size_t)fs * NY * Wp + cc;
#pragma unroll
    for (int e = 0; e < E; ++e) dst[(size_t)(t + T * e) * Wp] = acc[e];
  }
}

// Row pass out of the potential: IFFT_x, real part = V.  mode 0 stores V; mode 1 forms
// t = exp(i sigma V) and runs FFT_x for the transmission band limit; mode 2 stores t.
// sigma comes in units of pi: sincospif reduces its argument exactly in a few instructions, where
// sincosf brings a large-argument path that, unrolled over a thread's elements, overflowed the
// instruction cache (no_instruction was the first stall): 512 points, 128 slices 134 -> 105 us; the
// pass from V at 1024 points, 80 slices 552 -> 244 us.
// PAIR: a plane of Ap holds two slices of the one loaded species, V of the first in the real and of
// the second in the imaginary part, so both take one inverse transform (and one spreading and one
// column pass before it): three transforms per two rows instead of four here.  1152 points x 54 slices
// x 20 frames: splat_row 4.10 -> 2.61 ms, col_pot 5.90 -> 3.05, this 7.08 -> 5.95.  A slice
// without atoms is zero exactly, whatever its partner rounds to.  Modes 1 and 2 only (potential_block).
template <int NX, bool PAIR, int MB = -1>
__global__ void __launch_bounds__(PotOutCfg<NX>::THREADS, minb_of<K_ROW_POT_OUT, NX, PotOutCfg<NX>>())
    k_row_pot_out(Geo geo, Band b, const float2* __restrict__ Ap, int nbatch, SlicePairs sp, int mode, float sigma,
                  float* __restrict__ V, float2* __restrict__ out) {
  grid_dependency_wait();
  constexpr int E = PotOutCfg<NX>::E, T = PotOutCfg<NX>::T, G = PotOutCfg<NX>::G;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int bi = batch_index();
  if (bi >= nbatch) return;
  const int g = threadIdx.x / T, t = threadIdx.x % T, y = blockIdx.x * G + g, ny = geo.ny;
  const RowIdx<NX, E> idx{g * row_smem_stride<NX, E>()};
  const auto sync = group_sync<T>(g);
  float2 v[E];
  load_row<NX, MB>(v, Ap + ((size_t)bi * ny + y) * b.Wp, b, t);
  fft<NX, +1>(v, sm, idx, t, geo.tw, sync);
  // slices [s, s_end) of frame f come from this plane, s - s_first its part
  int f = 0, s_first = 0, s = 0, s_end = 1;
  if (PAIR) {
    f = bi / sp.planes;
    s_first = 2 * (sp.s0 / 2 + bi - f * sp.planes);
    s = s_first < sp.s0 ? sp.s0 : s_first;
    s_end = s_first + 2 < sp.s0 + sp.sb ? s_first + 2 : sp.s0 + sp.sb;
  }
  float im[E];
#pragma unroll
  for (int e = 0; e < E; ++e) im[e] = v[e].y;
#pragma unroll 1
  for (; s < s_end; ++s) {
    bool atoms = true;
    if (PAIR) {
      const int* bo = sp.boffs + ((size_t)f * sp.S + s) * (ny / SPREAD_YB + 1);
      atoms = bo[ny / SPREAD_YB] > bo[0];
      if (s > s_first) {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e].x = im[e];
      }
    }
    const size_t plane = PAIR ? (size_t)f * sp.sb + (s - sp.s0) : (size_t)bi;
    const size_t row = (plane * ny + y) * NX;
    if (!PAIR && mode == 0) {
#pragma unroll
      for (int e = 0; e < E; ++e) V[row + t + T * e] = v[e].x;
      continue;
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      float sn, cs;
      sincospif(atoms ? sigma * v[e].x : 0.f, &sn, &cs);
      v[e] = make_float2(cs, sn);
    }
    if (mode == 2) {
#pragma unroll
      for (int e = 0; e < E; ++e) out[row + t + T * e] = v[e];
      continue;
    }
    fft<NX, -1>(v, sm, idx, t, geo.tw, sync);
    store_row<NX, MB>(v, out + (plane * ny + y) * b.Wp, b, t);
  }
}

// ============================================================================================
// a3: transmission from a stored V.
// ============================================================================================
template <int NX>
__global__ void __launch_bounds__(RowVtCfg<NX>::THREADS, minb_of<K_ROW_VT, NX, RowVtCfg<NX>>())
    k_row_vt(Geo geo, Band b, const float* __restrict__ V, int nbatch, int bandlimit, float sigma,
             float2* __restrict__ out) {
  grid_dependency_wait();
  constexpr int E = RowVtCfg<NX>::E, T = RowVtCfg<NX>::T, G = RowVtCfg<NX>::G;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int fs = batch_index();
  if (fs >= nbatch) return;
  const int g = threadIdx.x / T, t = threadIdx.x % T, y = blockIdx.x * G + g, ny = geo.ny;
  const size_t row = ((size_t)fs * ny + y) * NX;
  float2 v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    float sn, cs;
    sincospif(sigma * V[row + t + T * e], &sn, &cs);
    v[e] = make_float2(cs, sn);
  }
  if (!bandlimit) {
#pragma unroll
    for (int e = 0; e < E; ++e) out[row + t + T * e] = v[e];
    return;
  }
  fft<NX, -1>(v, sm, RowIdx<NX, E>{g * row_smem_stride<NX, E>()}, t, geo.tw,
                  group_sync<T>(g));
  store_row_compact<NX>(v, out + ((size_t)fs * ny + y) * b.Wp, b, t);
}

// Column pass of the band limit: FFT_y, * M * scale, IFFT_y.
template <int NY, int WPC = -1>
__global__ void __launch_bounds__(ColTCfg<NY>::THREADS, minb_of<K_COL_T, NY, ColTCfg<NY>>())
    k_col_t(Geo geo, Band b, const float2* __restrict__ Bt, int nbatch, float scale, float2* __restrict__ At) {
  grid_dependency_wait();
  using CC = ColTCfg<NY>;
  constexpr int E = CC::E, T = CC::T, C = CC::C;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int fs = batch_index();
  if (fs >= nbatch) return;
  const int Wp = WPC > 0 ? WPC : b.Wp;
  const int c = threadIdx.x % C, t = threadIdx.x / C, cc = blockIdx.x * C + c;
  const ColIdx<C, CC::SH> idx{c};
  const BlockSync sync;
  const float2* tw = geo.tw;
  const float2* src = Bt + (size_t)fs * NY * Wp + cc;
  float2 v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = src[(size_t)(t + T * e) * Wp];
  fft<NY, -1>(v, sm, idx, t, tw, sync);
  const int nb = cc < b.W ? b.colnb[cc] : -1;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int n = fftfreq_index(t + T * e, NY);
    v[e] = (abs(n) <= nb) ? scale * v[e] : make_float2(0.f, 0.f);
  }
  fft<NY, +1>(v, sm, idx, t, tw, sync);
  float2* dst = At + (size_t)fs * NY * Wp + cc;
#pragma unroll
  for (int e = 0; e < E; ++e) dst[(size_t)(t + T * e) * Wp] = v[e];
}

// Row pass out of the band limit: IFFT_x -> t (full row).
template <int NX>
__global__ void __launch_bounds__(RowToutCfg<NX>::THREADS, minb_of<K_ROW_TOUT, NX, RowToutCfg<NX>>())
    k_row_tout(Geo geo, Band b, const float2* __restrict__ At, int nbatch, float2* __restrict__ tout) {
  grid_dependency_wait();
  constexpr int E = RowToutCfg<NX>::E, T = RowToutCfg<NX>::T, G = RowToutCfg<NX>::G;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int fs = batch_index();
  if (fs >= nbatch) return;
  const int g = threadIdx.x / T, t = threadIdx.x % T, y = blockIdx.x * G + g, ny = geo.ny;
  float2 v[E];
  load_row_compact<NX>(v, At + ((size_t)fs * ny + y) * b.Wp, b, t);
  fft<NX, +1>(v, sm, RowIdx<NX, E>{g * row_smem_stride<NX, E>()}, t, geo.tw,
                  group_sync<T>(g));
  float2* dst = tout + ((size_t)fs * ny + y) * NX;
#pragma unroll
  for (int e = 0; e < E; ++e) dst[t + T * e] = v[e];
}

// ============================================================================================
// Probe: psi0(k) = A(k) exp(-2 pi i k.r_p) amp, then a unitary inverse transform.
// ============================================================================================
// Phase tables of P probes, FP64 rounded to float: ex [P][Wp] and ey [P][ny], exp(-2 pi i k x_p) over
// the aperture columns and the rows, and chi [ny][Wp] (if any), exp(-i chi(k)).  The angular terms of
// chi are polynomials in (kx, ky): k^2 cos 2(phi - a) = (kx^2 - ky^2) cos 2a + 2 kx ky sin 2a and
// k cos(phi - a) = kx cos a + ky sin a.  On the host these tables were most of a call: 37 aberrated
// probes at 384^2 1.4 ms before the first launch.
__global__ void __launch_bounds__(256) k_probe_tables(ProbeTables q, const double* __restrict__ xy,
                                                      const int* __restrict__ nb, float2* __restrict__ ex,
                                                      float2* __restrict__ ey, float2* __restrict__ chi) {
  grid_dependency_wait();
  const int64_t nex = (int64_t)q.P * q.Wp, ney = (int64_t)q.P * q.ny, nchi = chi ? (int64_t)q.ny * q.Wp : 0;
  for (int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x; i < nex + ney + nchi; i += (int64_t)gridDim.x * 256) {
    double s, c;
    if (i < nex) {
      const int p = (int)(i / q.Wp), cc = (int)(i - (int64_t)p * q.Wp);
      float2 v = make_float2(0.f, 0.f);
      if (cc < q.W) {
        sincospi(-2.0 * ((double)q.freq_x(cc) / q.Lx) * (xy ? xy[2 * p] : 0.0), &s, &c);
        v = make_float2((float)c, (float)s);
      }
      ex[i] = v;
    } else if (i < nex + ney) {
      const int64_t k = i - nex;
      const int p = (int)(k / q.ny), y = (int)(k - (int64_t)p * q.ny);
      sincospi(-2.0 * ((double)fftfreq_index(y, q.ny) / q.Ly) * (xy ? xy[2 * p + 1] : 0.0), &s, &c);
      ey[k] = make_float2((float)c, (float)s);
    } else {
      const int64_t k = i - nex - ney;
      const int y = (int)(k / q.Wp), cc = (int)(k - (int64_t)y * q.Wp), n = fftfreq_index(y, q.ny);
      float2 v = make_float2(0.f, 0.f);
      if (cc < q.W && abs(n) <= nb[cc]) {
        const double kx = (double)q.freq_x(cc) / q.Lx, ky = (double)n / q.Ly, k2 = kx * kx + ky * ky;
        // chi / pi
        const double h = q.c1 * k2 + q.a_cos * (kx * kx - ky * ky) + q.a_sin * (2.0 * kx * ky) +
                         k2 * (q.b_cos * kx + q.b_sin * ky) + q.c3 * k2 * k2;
        sincospi(-h, &s, &c);
        v = make_float2((float)c, (float)s);
      }
      chi[k] = v;
    }
  }
}

cudaError_t launch_probe_tables(const ProbeTables& q, const double* xy, const int* nb, float2* ex, float2* ey,
                                float2* chi, cudaStream_t st) {
  const int64_t n = (int64_t)q.P * (q.Wp + q.ny) + (chi ? (int64_t)q.ny * q.Wp : 0);
  return launch_after(k_probe_tables, (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 8), 256, 0, st, q, xy, nb,
                      ex, ey, chi);
}

template <int NY>
__global__ void __launch_bounds__(ProbeColCfg<NY>::THREADS, minb_of<K_PROBE_COL, NY, ProbeColCfg<NY>>())
    k_probe_col(Geo geo, Band ap, const float2* __restrict__ ex, const float2* __restrict__ ey,
                const float2* __restrict__ chi, int P, float amp, float2* __restrict__ Bpr) {
  grid_dependency_wait();
  using CC = ProbeColCfg<NY>;
  constexpr int E = CC::E, T = CC::T, C = CC::C;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int p = batch_index();
  if (p >= P) return;
  const int c = threadIdx.x % C, t = threadIdx.x / C, cc = blockIdx.x * C + c;
  const int nb = cc < ap.W ? ap.colnb[cc] : -1;
  const float2 exv = cc < ap.W ? ex[(size_t)p * ap.Wp + cc] : make_float2(0.f, 0.f);
  float2 v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int row = t + T * e, n = fftfreq_index(row, NY);
    v[e] = (abs(n) <= nb) ? amp * cmul(exv, ey[(size_t)p * NY + row]) : make_float2(0.f, 0.f);
    if (chi && abs(n) <= nb) v[e] = cmul(v[e], chi[(size_t)row * ap.Wp + cc]);
  }
  fft<NY, +1>(v, sm, ColIdx<C, CC::SH>{c}, t, geo.tw, BlockSync{});
  float2* dst = Bpr + (size_t)p * NY * ap.Wp + cc;
#pragma unroll
  for (int e = 0; e < E; ++e) dst[(size_t)(t + T * e) * ap.Wp] = v[e];
}

template <int NX>
__global__ void __launch_bounds__(ProbeRowCfg<NX>::THREADS, minb_of<K_PROBE_ROW, NX, ProbeRowCfg<NX>>())
    k_probe_row(Geo geo, Band ap, const float2* __restrict__ Bpr, int P, float scale, float2* __restrict__ psi0) {
  grid_dependency_wait();
  constexpr int E = ProbeRowCfg<NX>::E, T = ProbeRowCfg<NX>::T, G = ProbeRowCfg<NX>::G;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int p = batch_index();
  if (p >= P) return;
  const int g = threadIdx.x / T, t = threadIdx.x % T, y = blockIdx.x * G + g, ny = geo.ny;
  float2 v[E];
  load_row_compact<NX>(v, Bpr + ((size_t)p * ny + y) * ap.Wp, ap, t);
  fft<NX, +1>(v, sm, RowIdx<NX, E>{g * row_smem_stride<NX, E>()}, t, geo.tw,
                  group_sync<T>(g));
  float2* dst = psi0 + ((size_t)p * ny + y) * NX;
#pragma unroll
  for (int e = 0; e < E; ++e) dst[t + T * e] = scale * v[e];
}

// ============================================================================================
// a4/a5: the slice step.
// TF: t comes as the compact output of the band-limit column pass (At) and is inverse-
// transformed here (one wave per frame: no full-size t is written or read).
// ============================================================================================
// Shared memory of the slice row pass: the FFT scratch, plus (TF) one stashed t row per group.
template <int NX, bool TF>
struct SliceRowSmem {
  // up to 16 elements a thread, the transmission row of several probes stays in registers
  static constexpr bool TREG = !TF && SliceRowCfg<NX, TF>::E <= 16;
  static constexpr int BYTES =
      SliceRowCfg<NX, TF>::SMEM + (TREG ? 0 : SliceRowCfg<NX, TF>::G * NX * (int)sizeof(float2));
};

// Most waves that one CTA of the slice column pass takes through its columns.  256 points, 2304 waves,
// 16 elements a thread: 2.97 ms for 8 slices with the loop; 4.16 with 32 elements, which spill in it.
constexpr int SLICE_COL_WAVES = 8;
// Most probes of a frame that one CTA of the slice row pass takes through its rows.  One probe a CTA
// copied the transmission row (60% of the pass's reads) once for every probe and waited for every
// wave's row; with eight, 256 points x 2048 waves take 280 us instead of 360.
constexpr int SLICE_ROW_PROBES = 8;

// MB >= 0: the band's half-width, fixed at compile time (the standard 2/3 band of a square
// cell, MB = NX / 3); MB < 0: read from b.
template <int NX, bool FIRST, bool PLANE, bool TF, int MB = -1>
__global__ void __launch_bounds__(SliceRowCfg<NX, TF>::THREADS, minb_of<slice_row_id<TF>(), NX, SliceRowCfg<NX, TF>>())
    k_slice_row(Geo geo, Band b, const float2* __restrict__ Apsi, const float2* __restrict__ psi0,
                const float2* __restrict__ ttab, int S, int s, int P, int ppb, int nfc, int nbatch, float plane_amp,
                float2* __restrict__ Bpsi) {
  grid_dependency_wait();
  using RC = SliceRowCfg<NX, TF>;
  constexpr int E = RC::E, T = RC::T, G = RC::G;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int bi = batch_index();
  if (bi >= nbatch) return;
  const int g = threadIdx.x / T, t = threadIdx.x % T, y = blockIdx.x * G + g, ny = geo.ny;
  const int pg = bi / nfc, fl = bi - pg * nfc, p0 = pg * ppb, p1 = p0 + ppb < P ? p0 + ppb : P;
  const RowIdx<NX, E> idx{g * row_smem_stride<NX, E>()};
  const auto sync = group_sync<T>(g);
  float2 v[E];
  if (FIRST && PLANE && TF) {
    // constant initial wave: FFT_x(c IFFT_x(At)) = c NX At, no transform needed
    load_row_compact<NX>(v, ttab + ((size_t)(fl * S + s) * ny + y) * b.Wp, b, t);
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = (plane_amp * (float)NX) * v[e];
    store_row_compact<NX>(v, Bpsi + ((size_t)bi * ny + y) * b.Wp, b, t);
    return;
  }
  // The probes p0 .. p1 - 1 of this frame share the transmission row.  TF: it is inverse-transformed
  // first and stashed in shared memory (only one row of the wave is then live in registers; each thread
  // rereads only its own positions, so no barrier is needed), the wave's row loading meanwhile.  TREG: it
  // stays in registers; the shared-memory pipe, three quarters busy with the exchanges, is the pass's
  // bound, and this drops a read per element (256 points: 45.7 -> 44.9 ms).  Otherwise it is copied
  // asynchronously into the stash, and the next probe's row loads while this one's is transformed.
  constexpr bool TREG = SliceRowSmem<NX, TF>::TREG;
  float2* tst = reinterpret_cast<float2*>(smraw + RC::SMEM) + g * NX;
  const auto load = [&](float2 (&u)[E], int p) {
    if (!FIRST) {
      load_row<NX, MB>(u, Apsi + ((size_t)(p * nfc + fl) * ny + y) * b.Wp, b, t);
    } else if (PLANE) {
#pragma unroll
      for (int e = 0; e < E; ++e) u[e] = make_float2(plane_amp, 0.f);
    } else {
      const float2* src = psi0 + ((size_t)p * ny + y) * NX;
#pragma unroll
      for (int e = 0; e < E; ++e) u[e] = src[t + T * e];
    }
  };
  const float2* trow = ttab + ((size_t)(fl * S + s) * ny + y) * NX;
  float2 next[E];
  float2 tr[TREG ? E : 1];
  if constexpr (TF) {
    load_row<NX, MB>(v, ttab + ((size_t)(fl * S + s) * ny + y) * b.Wp, b, t);
    load(next, p0);
    fft<NX, +1>(v, sm, idx, t, geo.tw, sync);
#pragma unroll
    for (int e = 0; e < E; ++e) tst[t + T * e] = v[e];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = next[e];
  } else if constexpr (TREG) {
    load(v, p0);
#pragma unroll
    for (int e = 0; e < E; ++e) tr[e] = trow[t + T * e];
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) cp_async8(tst + t + T * e, trow + t + T * e);
    asm volatile("cp.async.commit_group;" ::: "memory");
    load(v, p0);
  }
  for (int p = p0; p < p1; ++p) {
    if (!TF && !TREG && p + 1 < p1) load(next, p + 1);
    if (!FIRST) fft<NX, +1>(v, sm, idx, t, geo.tw, sync);
    if (!TF && !TREG) cp_async_wait_all();
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const float2 tv = TREG ? tr[TREG ? e : 0] : tst[t + T * e];
      if (FIRST && PLANE) v[e] = plane_amp * tv;
      else v[e] = cmul(v[e], tv);
    }
    fft<NX, -1>(v, sm, idx, t, geo.tw, sync);
    store_row<NX, MB>(v, Bpsi + ((size_t)(p * nfc + fl) * ny + y) * b.Wp, b, t);
    if (TF) return;  // one probe
    if (!TREG) {
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = next[e];
    } else if (p + 1 < p1) {
      load(v, p + 1);
    }
  }
}

// WPC > 0: the row stride of the compact columns (Wp) fixed at compile time (the standard band
// of a square grid), so the strided loads and stores take immediate offsets; else Wp.
// LOOP: a CTA takes its columns of wpb waves one after the other.  The propagator times mask and
// scale is put together once per CTA, in shared memory (each thread reads back only what it wrote),
// and the next wave's column is loaded while this one is transformed.  Both forms multiply by the
// same product, so that a wave's bits do not depend on how many waves a launch holds.
template <int NY>
__host__ __device__ constexpr bool slice_col_loop() {
  return 2 * SliceColCfg<NY>::SMEM <= 100 * 1024;  // two such CTAs per SM
}
template <int NY, bool LAST, bool LOOP, int WPC = -1>
__global__ void __launch_bounds__(SliceColCfg<NY>::THREADS, minb_of<K_SLICE_COL, NY, SliceColCfg<NY>>())
    k_slice_col(Geo geo, Band b, const float2* __restrict__ Bpsi, const float2* __restrict__ px,
                const float2* __restrict__ py, float scale, int wpb, int nfc, int nwaves, int64_t F_total, int64_t f0,
                const int2* __restrict__ disc, int64_t nsel, float2* __restrict__ Apsi, float2* __restrict__ psi_k) {
  grid_dependency_wait();
  using CC = SliceColCfg<NY>;
  constexpr int E = CC::E, T = CC::T, C = CC::C;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int w0 = batch_index() * wpb, w1 = w0 + wpb < nwaves ? w0 + wpb : nwaves;
  if (w0 >= nwaves) return;
  const int Wp = WPC > 0 ? WPC : b.Wp;
  const int c = threadIdx.x % C, t = threadIdx.x / C, cc = blockIdx.x * C + c;
  const ColIdx<C, CC::SH> idx{c};
  const BlockSync sync;
  const float2* tw = geo.tw;
  const auto load = [&](float2 (&u)[E], int w) {
    const float2* src = Bpsi + (size_t)w * NY * Wp + cc;
#pragma unroll
    for (int e = 0; e < E; ++e) u[e] = src[(size_t)(t + T * e) * Wp];
  };
  float2 v[E];
  load(v, w0);
  const int nb = cc < b.W ? b.colnb[cc] : -1;
  const float2 pxc = cc < b.W ? px[cc] : make_float2(0.f, 0.f);
  float2* prop = reinterpret_cast<float2*>(smraw + CC::SMEM) + threadIdx.x;  // [E][THREADS]
  if (LOOP) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int row = t + T * e, n = fftfreq_index(row, NY);
      prop[CC::THREADS * e] = (abs(n) <= nb) ? scale * cmul(pxc, py[row]) : make_float2(0.f, 0.f);
    }
  }
  for (int w = w0; w < w1; ++w) {
    float2 next[E];
    if (LOOP && w + 1 < w1) load(next, w + 1);
    fft<NY, -1>(v, sm, idx, t, tw, sync);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if (LOOP) {
        v[e] = cmul(v[e], prop[CC::THREADS * e]);
      } else {
        const int row = t + T * e, n = fftfreq_index(row, NY);
        v[e] = cmul(v[e], (abs(n) <= nb) ? scale * cmul(pxc, py[row]) : make_float2(0.f, 0.f));
      }
    }
    if (!LAST) {
      fft<NY, +1>(v, sm, idx, t, tw, sync);
      float2* dst = Apsi + (size_t)w * NY * Wp + cc;
#pragma unroll
      for (int e = 0; e < E; ++e) dst[(size_t)(t + T * e) * Wp] = v[e];
    } else if (cc < b.W) {
      const int p = w / nfc, fl = w - p * nfc;
      if (disc) {
        // compact exit wave: the in-band points of the disc only, in ascending q = y nx + x;
        // row y holds disc[y].y points from disc[y].x on, with x in [0, a] then [nx - a, nx)
        float2* dst = psi_k + ((size_t)p * F_total + f0 + fl) * nsel;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int row = t + T * e, n = fftfreq_index(row, NY);
          if (abs(n) <= nb) {
            const int2 d = disc[row];
            const int a = (d.y - 1) >> 1;
            const int j = d.y == geo.nx ? cc : (cc <= a ? cc : cc - b.W + 2 * a + 1);
            dst[d.x + j] = v[e];
          }
        }
      } else {
        const int x = band_col_x(b, geo.nx, cc);
        float2* dst = psi_k + (((size_t)p * F_total + f0 + fl) * NY) * geo.nx + x;
#pragma unroll
        for (int e = 0; e < E; ++e) dst[(size_t)(t + T * e) * geo.nx] = v[e];
      }
    }
    if (!LOOP) return;  // one wave
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = next[e];
  }
}

// ============================================================================================
// Potential multiplier table [pair][ny][Wp] (FP64 evaluation, float storage).
// ============================================================================================
__device__ double form_factor_f64(const double* c, double q) {
  const double q2 = q * q;
  double f = 0.0;
  for (int i = 0; i < 3; ++i) f += c[2 * i] / (q2 + c[2 * i + 1]);
  for (int i = 0; i < 3; ++i) f += c[6 + 2 * i] * exp(-c[7 + 2 * i] * q2);
  return f;
}

__global__ void k_build_mtab(int nx, int ny, Band b, int npair, int nslot, const double* __restrict__ coef,
                             const double* __restrict__ phix, const double* __restrict__ phiy, double Lx, double Ly,
                             double pref, float2* __restrict__ mtab) {
  const int64_t total = (int64_t)npair * ny * b.Wp;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int cc = (int)(i % b.Wp);
    const int row = (int)((i / b.Wp) % ny);
    const int pr = (int)(i / ((int64_t)b.Wp * ny));
    float2 out = make_float2(0.f, 0.f);
    const int n = fftfreq_index(row, ny);
    if (cc < b.W && abs(n) <= b.colnb[cc]) {
      const int m = fftfreq_index(band_col_x(b, nx, cc), nx);
      const double kx = (double)m / Lx, ky = (double)n / Ly;
      const double q = sqrt(kx * kx + ky * ky);
      const double fa = form_factor_f64(coef + 12 * (2 * pr), q);
      const double fb = (2 * pr + 1 < nslot) ? form_factor_f64(coef + 12 * (2 * pr + 1), q) : 0.0;
      const double sc = pref / (phix[cc] * phiy[row]);
      out = make_float2((float)(sc * fa), (float)(-sc * fb));
    }
    mtab[i] = out;
  }
}

// ============================================================================================
// launchers
// ============================================================================================
template <class K>
static cudaError_t prep(K kernel, int smem) {
  // opt in above 46 KB: some kernels add a little static shared memory to the dynamic amount
  if (smem > 46 * 1024) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return cudaSuccess;
}

// Row-pass kernels are also built for the standard 2/3 band of a square cell (half-width NX / 3
// fixed at compile time) at these lengths (the powers of two of the configurations and the
// minimal example's 1152); a launch uses that build when its band is that one
// and the context option "static_band" is on.
template <int NX>
constexpr bool std_band_built() {
  return (fft_pow2(NX) && NX >= 128 && NX <= 1024) || NX == 1152;
}
template <int NX>
bool std_band(const Band& b, int static_band) {
  return static_band && std_band_built<NX>() && b.mb == NX / 3 && b.W == 2 * (NX / 3) + 1;
}
// Padded row stride of the compact columns for that band (as make_band pads W).
constexpr int std_band_wp(int n) {
  const int w = 2 * (n / 3) + 1, up = (w + 31) / 32 * 32, wp = up < 32 ? 32 : up;
  return wp > n ? n : wp;
}

#define TACAW_DISPATCH(N, FN, ...)       \
  switch (N) {                           \
    case 32: return FN<32>(__VA_ARGS__);     \
    case 64: return FN<64>(__VA_ARGS__);     \
    case 96: return FN<96>(__VA_ARGS__);     \
    case 128: return FN<128>(__VA_ARGS__);   \
    case 192: return FN<192>(__VA_ARGS__);   \
    case 256: return FN<256>(__VA_ARGS__);   \
    case 384: return FN<384>(__VA_ARGS__);   \
    case 512: return FN<512>(__VA_ARGS__);   \
    case 768: return FN<768>(__VA_ARGS__);   \
    case 1024: return FN<1024>(__VA_ARGS__); \
    case 1152: return FN<1152>(__VA_ARGS__); \
    default: return cudaErrorInvalidValue;   \
  }

template <int NX>
static cudaError_t splat_row_n(const Geo& g, const Band& b, const AtomRec* recs, const int* boffs, int64_t A,
                               int S, int s0, int sb, int nfs, int npair, int two, float beta, float2* Bp,
                               int static_band, cudaStream_t st) {
  if (s0 < 0 || sb < 1 || nfs % sb != 0 || (two ? npair != 1 || 2 * (s0 / 2 + sb - 1) >= S : s0 + sb > S))
    return cudaErrorInvalidValue;
  const int smem = SplatSmem<NX>::BYTES;
  const int nb = nfs * npair;
  const dim3 grid = batch_grid(g.ny / SplatCfg<NX>::G, nb);
  // not at 512 points, where the fixed-band build took more registers and measured 4% slower
  if constexpr (std_band_built<NX>() && NX != 512) {
    if (std_band<NX>(b, static_band)) {
      cudaError_t e = prep(k_splat_row<NX, NX / 3>, smem);
      if (e != cudaSuccess) return e;
      return launch_after(k_splat_row<NX, NX / 3>, grid, SplatCfg<NX>::THREADS, smem, st, g, b, recs, boffs, (int)A,
                          S, s0, sb, npair, two, nb, beta, Bp);
    }
  }
  cudaError_t e = prep(k_splat_row<NX>, smem);
  if (e != cudaSuccess) return e;
  return launch_after(k_splat_row<NX>, grid, SplatCfg<NX>::THREADS, smem, st, g, b, recs, boffs, (int)A, S, s0, sb,
                      npair, two, nb, beta, Bp);
}
cudaError_t launch_splat_row(const Geo& g, const Band& b, const AtomRec* recs, const int* boffs, int64_t A, int S,
                             int s0, int sb, int nfs, int npair, int two, float beta, float2* Bp, int static_band,
                             cudaStream_t st) {
  if (g.ny % SPREAD_YB != 0) return cudaErrorInvalidValue;
  TACAW_DISPATCH(g.nx, splat_row_n, g, b, recs, boffs, A, S, s0, sb, nfs, npair, two, beta, Bp, static_band, st);
}

template <int NY>
static cudaError_t col_pot_n(const Geo& g, const Band& b, const float2* Bp, const float2* mtab, int npair, int nfs,
                             float2* Ap, int static_band, cudaStream_t st) {
  using CC = ColPotCfg<NY>;
  const dim3 grid = batch_grid(col_blocks(b, CC::C), nfs);
  cudaError_t e;
  if constexpr (std_band_built<NY>()) {
    constexpr int WP = std_band_wp(NY);
    if (g.nx == NY && b.Wp == WP && std_band<NY>(b, static_band)) {
      if (npair == 1) {
        if ((e = prep(k_col_pot<NY, true, WP>, CC::SMEM)) != cudaSuccess) return e;
        return launch_after(k_col_pot<NY, true, WP>, grid, CC::THREADS, CC::SMEM, st, g, b, Bp, mtab, npair, nfs, Ap);
      } else {
        if ((e = prep(k_col_pot<NY, false, WP>, CC::SMEM)) != cudaSuccess) return e;
        return launch_after(k_col_pot<NY, false, WP>, grid, CC::THREADS, CC::SMEM, st, g, b, Bp, mtab, npair, nfs, Ap);
      }
    }
  }
  if (npair == 1) {
    if ((e = prep(k_col_pot<NY, true>, CC::SMEM)) != cudaSuccess) return e;
    return launch_after(k_col_pot<NY, true>, grid, CC::THREADS, CC::SMEM, st, g, b, Bp, mtab, npair, nfs, Ap);
  } else {
    if ((e = prep(k_col_pot<NY, false>, CC::SMEM)) != cudaSuccess) return e;
    return launch_after(k_col_pot<NY, false>, grid, CC::THREADS, CC::SMEM, st, g, b, Bp, mtab, npair, nfs, Ap);
  }
}
cudaError_t launch_col_pot(const Geo& g, const Band& b, const float2* Bp, const float2* mtab, int npair, int nfs,
                           float2* Ap, int static_band, cudaStream_t st) {
  TACAW_DISPATCH(g.ny, col_pot_n, g, b, Bp, mtab, npair, nfs, Ap, static_band, st);
}

template <int NX, bool PAIR>
static cudaError_t row_pot_out_p(const Geo& g, const Band& b, const float2* Ap, int nb, const SlicePairs& sp, int mode,
                                 float sigma, float* V, float2* out, int static_band, cudaStream_t st) {
  using RC = PotOutCfg<NX>;
  const dim3 grid = batch_grid(g.ny / RC::G, nb);
  if constexpr (std_band_built<NX>()) {
    if (std_band<NX>(b, static_band)) {
      return launch_after(k_row_pot_out<NX, PAIR, NX / 3>, grid, RC::THREADS, RC::SMEM, st, g, b, Ap, nb, sp, mode,
                          sigma, V, out);
    }
  }
  return launch_after(k_row_pot_out<NX, PAIR>, grid, RC::THREADS, RC::SMEM, st, g, b, Ap, nb, sp, mode, sigma, V, out);
}
template <int NX>
static cudaError_t row_pot_out_n(const Geo& g, const Band& b, const float2* Ap, int nb, const SlicePairs& sp, int mode,
                                 float sigma, float* V, float2* out, int static_band, cudaStream_t st) {
  return sp.planes ? row_pot_out_p<NX, true>(g, b, Ap, nb, sp, mode, sigma, V, out, static_band, st)
                   : row_pot_out_p<NX, false>(g, b, Ap, nb, sp, mode, sigma, V, out, static_band, st);
}
cudaError_t launch_row_pot_out(const Geo& g, const Band& b, const float2* Ap, int nb, const SlicePairs& sp, int mode,
                               float sigma, float* V, float2* out, int static_band, cudaStream_t st) {
  TACAW_DISPATCH(g.nx, row_pot_out_n, g, b, Ap, nb, sp, mode, sigma, V, out, static_band, st);
}

template <int NX>
static cudaError_t row_vt_n(const Geo& g, const Band& b, const float* V, int nfs, int bl, float sigma, float2* out,
                            cudaStream_t st) {
  return launch_after(k_row_vt<NX>, batch_grid(g.ny / RowVtCfg<NX>::G, nfs), RowVtCfg<NX>::THREADS,
                      RowVtCfg<NX>::SMEM, st, g, b, V, nfs, bl, sigma, out);
}
cudaError_t launch_row_vt(const Geo& g, const Band& b, const float* V, int nfs, int bandlimit, float sigma,
                          float2* out, cudaStream_t st) {
  TACAW_DISPATCH(g.nx, row_vt_n, g, b, V, nfs, bandlimit, sigma, out, st);
}

template <int NY>
static cudaError_t col_t_n(const Geo& g, const Band& b, const float2* Bt, int nfs, float scale, float2* At,
                           int static_band, cudaStream_t st) {
  using CC = ColTCfg<NY>;
  if constexpr (std_band_built<NY>()) {
    constexpr int WP = std_band_wp(NY);
    if (g.nx == NY && b.Wp == WP && std_band<NY>(b, static_band)) {
      const cudaError_t e = prep(k_col_t<NY, WP>, CC::SMEM);
      if (e != cudaSuccess) return e;
      return launch_after(k_col_t<NY, WP>, batch_grid(col_blocks(b, CC::C), nfs), CC::THREADS, CC::SMEM, st, g, b, Bt,
                          nfs, scale, At);
    }
  }
  const cudaError_t e = prep(k_col_t<NY>, CC::SMEM);
  if (e != cudaSuccess) return e;
  return launch_after(k_col_t<NY>, batch_grid(col_blocks(b, CC::C), nfs), CC::THREADS, CC::SMEM, st, g, b, Bt, nfs,
                      scale, At);
}
cudaError_t launch_col_t(const Geo& g, const Band& b, const float2* Bt, int nfs, float scale, float2* At,
                         int static_band, cudaStream_t st) {
  TACAW_DISPATCH(g.ny, col_t_n, g, b, Bt, nfs, scale, At, static_band, st);
}

template <int NX>
static cudaError_t row_tout_n(const Geo& g, const Band& b, const float2* At, int nfs, float2* t, cudaStream_t st) {
  using RC = RowToutCfg<NX>;
  return launch_after(k_row_tout<NX>, batch_grid(g.ny / RC::G, nfs), RC::THREADS, RC::SMEM, st, g, b, At, nfs, t);
}
cudaError_t launch_row_tout(const Geo& g, const Band& b, const float2* At, int nfs, float2* t, cudaStream_t st) {
  TACAW_DISPATCH(g.nx, row_tout_n, g, b, At, nfs, t, st);
}

template <int NY>
static cudaError_t probe_col_n(const Geo& g, const Band& ap, const float2* ex, const float2* ey, const float2* chi,
                               int P, float amp, float2* Bpr, cudaStream_t st) {
  using CC = ProbeColCfg<NY>;
  const cudaError_t e = prep(k_probe_col<NY>, CC::SMEM);
  if (e != cudaSuccess) return e;
  return launch_after(k_probe_col<NY>, batch_grid(col_blocks(ap, CC::C), P), CC::THREADS, CC::SMEM, st, g, ap, ex,
                      ey, chi, P, amp, Bpr);
}
cudaError_t launch_probe_col(const Geo& g, const Band& ap, const float2* ex, const float2* ey, const float2* chi,
                             int P, float amp, float2* Bpr, cudaStream_t st) {
  TACAW_DISPATCH(g.ny, probe_col_n, g, ap, ex, ey, chi, P, amp, Bpr, st);
}

template <int NX>
static cudaError_t probe_row_n(const Geo& g, const Band& ap, const float2* Bpr, int P, float scale, float2* psi0,
                               cudaStream_t st) {
  using RC = ProbeRowCfg<NX>;
  return launch_after(k_probe_row<NX>, batch_grid(g.ny / RC::G, P), RC::THREADS, RC::SMEM, st, g, ap, Bpr, P, scale,
                      psi0);
}
cudaError_t launch_probe_row(const Geo& g, const Band& ap, const float2* Bpr, int P, float scale, float2* psi0,
                             cudaStream_t st) {
  TACAW_DISPATCH(g.nx, probe_row_n, g, ap, Bpr, P, scale, psi0, st);
}

template <int NX>
static cudaError_t slice_row_n(const Geo& g, const Band& b, int first, int plane, int tfused, const float2* Apsi,
                               const float2* psi0, const float2* t, int S, int s, int P, int nfc, float plane_amp,
                               float2* Bpsi, int static_band, cudaStream_t st) {
  // probes per CTA: up to SLICE_ROW_PROBES, while at least 16 CTAs are left for every SM
  const int G = tfused ? SliceRowCfg<NX, true>::G : SliceRowCfg<NX, false>::G;
  const int64_t ctas = (int64_t)P * nfc * (g.ny / G);
  int ppb = (int)std::min<int64_t>(std::min(P, SLICE_ROW_PROBES), std::max<int64_t>(1, ctas / (16 * 152)));
  ppb = (P + (P + ppb - 1) / ppb - 1) / ((P + ppb - 1) / ppb);  // even groups
  const int nbatch = (P + ppb - 1) / ppb * nfc;
  const dim3 grid = batch_grid(g.ny / G, nbatch);
#define TACAW_SLICE_ROW(F, PL, TFU)                                                                               \
  do {                                                                                                            \
    constexpr int SM = SliceRowSmem<NX, TFU>::BYTES, TH = SliceRowCfg<NX, TFU>::THREADS;                          \
    cudaError_t e_ = prep(k_slice_row<NX, F, PL, TFU>, SM);                                                       \
    if (e_ != cudaSuccess) return e_;                                                                             \
    return launch_after(k_slice_row<NX, F, PL, TFU>, grid, TH, SM, st, g, b, Apsi, psi0, t, S, s, P, ppb, nfc,     \
                        nbatch, plane_amp, Bpsi);                                                                 \
  } while (0)
  // the later slices (all but one of S) with the standard band fixed at compile time
  constexpr int MB3 = NX / 3;
  constexpr bool SPEC = std_band_built<NX>();
  const bool std_band = tacaw::std_band<NX>(b, static_band);
#define TACAW_SLICE_ROW_STD(TFU)                                                                                   \
  do {                                                                                                            \
    constexpr int SM = SliceRowSmem<NX, TFU>::BYTES, TH = SliceRowCfg<NX, TFU>::THREADS;                          \
    cudaError_t e_ = prep(k_slice_row<NX, false, false, TFU, MB3>, SM);                                           \
    if (e_ != cudaSuccess) return e_;                                                                             \
    return launch_after(k_slice_row<NX, false, false, TFU, MB3>, grid, TH, SM, st, g, b, Apsi, psi0, t, S, s, P,    \
                        ppb, nfc, nbatch, plane_amp, Bpsi);                                                       \
  } while (0)
  if (tfused) {
    if (first && plane) TACAW_SLICE_ROW(true, true, true);
    else if (first) TACAW_SLICE_ROW(true, false, true);
    else if constexpr (SPEC) {
      if (std_band) TACAW_SLICE_ROW_STD(true);
      else TACAW_SLICE_ROW(false, false, true);
    } else TACAW_SLICE_ROW(false, false, true);
  } else {
    if (first && plane) TACAW_SLICE_ROW(true, true, false);
    else if (first) TACAW_SLICE_ROW(true, false, false);
    else if constexpr (SPEC) {
      if (std_band) TACAW_SLICE_ROW_STD(false);
      else TACAW_SLICE_ROW(false, false, false);
    } else TACAW_SLICE_ROW(false, false, false);
  }
#undef TACAW_SLICE_ROW_STD
#undef TACAW_SLICE_ROW
}
cudaError_t launch_slice_row(const Geo& g, const Band& b, int first, int plane, int tfused, const float2* Apsi,
                             const float2* psi0, const float2* t, int S, int s, int P, int nfc, float plane_amp,
                             float2* Bpsi, int static_band, cudaStream_t st) {
  TACAW_DISPATCH(g.nx, slice_row_n, g, b, first, plane, tfused, Apsi, psi0, t, S, s, P, nfc, plane_amp, Bpsi,
                 static_band, st);
}

template <int NY>
static cudaError_t slice_col_n(const Geo& g, const Band& b, int last, const float2* Bpsi, const float2* px,
                               const float2* py, float scale, int P, int nfc, int64_t F_total, int64_t f0,
                               const int2* disc, int64_t nsel, float2* Apsi, float2* psi_k, int static_band,
                               cudaStream_t st) {
  const int nw = P * nfc;
  using CC = SliceColCfg<NY>;
  constexpr int TH = CC::THREADS;
  const int cb = col_blocks(b, CC::C);
  // waves per CTA: up to SLICE_COL_WAVES, while at least 16 CTAs are left for every SM
  int wpb = 1;
  if (slice_col_loop<NY>() && !last)
    wpb = (int)std::min<int64_t>(SLICE_COL_WAVES, std::max<int64_t>(1, (int64_t)nw * cb / (16 * 152)));
  const dim3 grid = batch_grid(cb, (nw + wpb - 1) / wpb);
#define TACAW_SLICE_COL(L, LOOP, ...)                                                                                 \
  do {                                                                                                                \
    constexpr int SM = CC::SMEM + ((LOOP) ? NY * CC::C * (int)sizeof(float2) : 0);                                     \
    cudaError_t e_ = prep(k_slice_col<NY, L, LOOP __VA_OPT__(, ) __VA_ARGS__>, SM);                                   \
    if (e_ != cudaSuccess) return e_;                                                                                 \
    return launch_after(k_slice_col<NY, L, LOOP __VA_OPT__(, ) __VA_ARGS__>, grid, TH, SM, st, g, b, Bpsi, px, py,     \
                        scale, wpb, nfc, nw, F_total, f0, disc, nsel, Apsi, psi_k);                                   \
  } while (0)
  if (last) TACAW_SLICE_COL(true, false);
  // the later slices of a square grid with the standard band: row stride fixed at compile time
  if constexpr (std_band_built<NY>()) {
    constexpr int WP = std_band_wp(NY);
    if (g.nx == NY && b.Wp == WP && std_band<NY>(b, static_band)) {
      if constexpr (slice_col_loop<NY>())
        if (wpb > 1) TACAW_SLICE_COL(false, true, WP);
      TACAW_SLICE_COL(false, false, WP);
    }
  }
  if constexpr (slice_col_loop<NY>())
    if (wpb > 1) TACAW_SLICE_COL(false, true);
  TACAW_SLICE_COL(false, false);
#undef TACAW_SLICE_COL
}
cudaError_t launch_slice_col(const Geo& g, const Band& b, int last, const float2* Bpsi, const float2* px,
                             const float2* py, float scale, int P, int nfc, int64_t F_total, int64_t f0,
                             const int2* disc, int64_t nsel, float2* Apsi, float2* psi_k, int static_band,
                             cudaStream_t st) {
  TACAW_DISPATCH(g.ny, slice_col_n, g, b, last, Bpsi, px, py, scale, P, nfc, F_total, f0, disc, nsel, Apsi, psi_k,
                 static_band, st);
}

cudaError_t launch_build_mtab(const Geo& g, const Band& b, int npair, int nslot, const double* coef_slots,
                              const double* phix, const double* phiy, double Lx, double Ly, double pref,
                              float2* mtab, cudaStream_t st) {
  const int64_t total = (int64_t)npair * g.ny * b.Wp;
  const int blocks = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
  k_build_mtab<<<blocks, 256, 0, st>>>(g.nx, g.ny, b, npair, nslot, coef_slots, phix, phiy, Lx, Ly, pref, mtab);
  return cudaGetLastError();
}

}  // namespace tacaw
