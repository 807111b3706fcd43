// Exact binning of samples into per-pixel FP64 sums for the set-up and the operators (weight
// blocks, P^T of a caller's timestream, the allocation-free binned map): sums over runs of
// consecutive samples on one pixel first, one FP64 reduction per run and sum afterwards.
//
// What bounds it: a reduction per sample and sum saturates the L2's atomic units (12 per
// sample for the weight blocks: 1.90 ms for 8 x 2^22 samples), and FP64 arithmetic runs on a
// pipe of about two lanes per SM and clock.  So the runs of a tile of 1024 samples are listed
// by warp ballots, a thread sums one run (5 to 8 FP64 instructions a sample, products and sums
// contracted), and the finished sums are handed out again one (run, sum) per lane, so that a
// warp's reductions cover the consecutive words of two to ten pixels instead of 32 scattered
// ones.  Measured on 512^2 IQU rasters at 4 samples per pixel: weight blocks of 8 x 2^22
// samples 1900 -> 652 us (9.96 M FP64 warp instructions, 0.5 ms of that pipe), P^T 425 -> 289 us,
// binned map of 2 x 2^22 samples 349 -> 181 us.
#pragma once

#include "mm_internal.cuh"

namespace mm {

// Exact FP32 -> FP64 widening that keeps subnormal inputs (f32_to_f64 flushes them).
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f) & 0x7fffffffu;
  return u - 1u < 0x7fffffu ? (double)f : f32_to_f64(f);
}

// One weight of sample s, FP32 or FP16 storage.
__device__ __forceinline__ float load_w(const void* w, int half_w, int64_t s) {
  return half_w ? __half2float(static_cast<const __half*>(w)[s]) : static_cast<const float*>(w)[s];
}

constexpr int kBinTile = 1024, kBinThreads = 256;

// Op: NF float streams per sample (load), NV sums per run (add), NO outputs per run (emit).
// Samples [n0, n1); samples with a pixel outside [0, n_pix) are skipped.  Op::tile(first,
// last, shared) prepares per-tile state (every thread, before a barrier); Op::cut(i) marks a tile
// position that starts a run whatever its pixel.
template <class Op>
__global__ void __launch_bounds__(kBinThreads) k_run_bin(Op op, const int32_t* __restrict__ pix,
                                                         int64_t n0, int64_t n1, int64_t n_pix) {
  constexpr int NF = Op::NF, NV = Op::NV, NO = Op::NO, W = kBinThreads / 32;
  constexpr int SV = NV | 1;   // odd stride: the sums of neighbouring runs on different banks
  __shared__ int s_pix[kBinTile];
  __shared__ float s_f[NF > 0 ? NF : 1][kBinTile];
  __shared__ uint16_t s_run[kBinTile];     // first position | (length - 1) << 11, valid runs only
  static_assert(kBinTile <= 2048, "11 bits of position");
  __shared__ double s_val[kBinThreads * SV];
  __shared__ int s_cnt[W];
  __shared__ double s_op[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t base = n0 + (int64_t)blockIdx.x * kBinTile;
  const int cnt = n1 - base < kBinTile ? (int)(n1 - base) : kBinTile;
  op.tile(base, base + cnt - 1, s_op);
#pragma unroll
  for (int k = 0; k < kBinTile / kBinThreads; ++k) {
    const int i = threadIdx.x + k * kBinThreads;
    if (i < cnt) {
      s_pix[i] = pix[base + i];
#pragma unroll
      for (int f = 0; f < NF; ++f) s_f[f][i] = op.load(f, base + i);
    }
  }
  __syncthreads();
  // run starts: warp w lists positions [256 w, 256 w + 256) in rounds of 32; position 0 of a
  // round always starts a run, so a run lies within its round (and has at most 32 samples)
  constexpr int R = kBinTile / kBinThreads;
  unsigned head[R], keep[R];
  int mine = 0;
#pragma unroll
  for (int k = 0; k < R; ++k) {
    const int i = warp * (32 * R) + 32 * k + lane;
    const int p = i < cnt ? s_pix[i] : -1;
    const bool h = lane == 0 || i >= cnt || p != s_pix[i - 1] || op.cut(i);
    head[k] = __ballot_sync(0xffffffffu, h);
    keep[k] = __ballot_sync(0xffffffffu, h && i < cnt && p >= 0 && p < n_pix);
    mine += __popc(keep[k]);
  }
  if (lane == 0) s_cnt[warp] = mine;
  __syncthreads();
  int at = 0, nrun = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const int c = s_cnt[w];
    at += w < warp ? c : 0;
    nrun += c;
  }
#pragma unroll
  for (int k = 0; k < R; ++k) {
    if ((keep[k] >> lane) & 1u) {
      const unsigned later = lane == 31 ? 0u : head[k] >> (lane + 1);
      const int len = later ? __ffs(later) : 32 - lane;
      s_run[at + __popc(keep[k] & ((1u << lane) - 1u))] =
          (uint16_t)((warp * (32 * R) + 32 * k + lane) | (len - 1) << 11);
    }
    at += __popc(keep[k]);
  }
  __syncthreads();
  for (int r0 = 0; r0 < nrun; r0 += kBinThreads) {
    const int nb = nrun - r0 < kBinThreads ? nrun - r0 : kBinThreads;
    if ((int)threadIdx.x < nb) {
      const int e = s_run[r0 + threadIdx.x], a = e & 2047, b = a + (e >> 11) + 1;
      double v[NV];
#pragma unroll
      for (int j = 0; j < NV; ++j) v[j] = 0.0;
      for (int i = a; i < b; ++i) {
        float f[NF > 0 ? NF : 1];
#pragma unroll
        for (int j = 0; j < NF; ++j) f[j] = s_f[j][i];
        op.add(v, f);
      }
      op.close(v, b - a);
#pragma unroll
      for (int j = 0; j < NV; ++j) s_val[threadIdx.x * SV + j] = v[j];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nb * NO; t += kBinThreads) {
      const int r = t / NO, o = t - r * NO;
      const int a = s_run[r0 + r] & 2047;
      op.emit(s_pix[a], o, s_val + r * SV, base + a, s_op);
    }
    __syncthreads();
  }
}

template <class Op>
static cudaError_t launch_run_bin(const Op& op, const int32_t* pix, int64_t n0, int64_t n1,
                                  int64_t n_pix, cudaStream_t st) {
  if (n1 <= n0) return cudaSuccess;
  k_run_bin<Op><<<(unsigned)((n1 - n0 + kBinTile - 1) / kBinTile), kBinThreads, 0, st>>>(op, pix, n0, n1, n_pix);
  return cudaGetLastError();
}

// P^T t into interleaved [n_pix][NC] sums.
template <int NC>
struct BinPT {
  static constexpr int NF = NC == 3 ? 3 : 1, NV = NC, NO = NC;
  const float* tod;
  const void *cosw, *sinw;
  int half_w;
  double* out;
  __device__ void tile(int64_t, int64_t, double*) {}
  __device__ bool cut(int) const { return false; }
  __device__ float load(int f, int64_t s) const {
    return f == 0 ? tod[s] : load_w(f == 1 ? cosw : sinw, half_w, s);
  }
  __device__ void add(double* v, const float* f) const {
    const double t = widen(f[0]);
    v[0] += t;
    if constexpr (NC == 3) {
      v[1] = fma(t, widen(f[1]), v[1]);
      v[2] = fma(t, widen(f[2]), v[2]);
    }
  }
  __device__ void close(double*, int) const {}
  __device__ void emit(int p, int o, const double* v, int64_t, const double*) const {
    atomicAdd(out + (int64_t)NC * p + o, v[o]);
  }
};

// Normal-equation sums of the unit-weight binned map, kStride doubles per pixel: hits, then
// (IQU) c, s, cc, cs, ss, d, dc, ds or (T) d.
template <int NC, int kStride>
struct BinNormal {
  static constexpr int NF = NC == 3 ? 3 : 1, NV = NC == 3 ? 9 : 2, NO = NV;
  const float* tod;
  const void *cosw, *sinw;
  int half_w;
  double* out;
  __device__ void tile(int64_t, int64_t, double*) {}
  __device__ bool cut(int) const { return false; }
  __device__ float load(int f, int64_t s) const {
    return f == 0 ? tod[s] : load_w(f == 1 ? cosw : sinw, half_w, s);
  }
  __device__ void add(double* v, const float* f) const {
    const double t = widen(f[0]);
    if constexpr (NC == 1) {
      v[1] += t;
    } else {
      const double c = widen(f[1]), w = widen(f[2]);
      v[1] += c;
      v[2] += w;
      v[3] = fma(c, c, v[3]);
      v[4] = fma(c, w, v[4]);
      v[5] = fma(w, w, v[5]);
      v[6] += t;
      v[7] = fma(t, c, v[7]);
      v[8] = fma(t, w, v[8]);
    }
  }
  __device__ void close(double* v, int len) const { v[0] = (double)len; }
  __device__ void emit(int p, int o, const double* v, int64_t, const double*) const {
    atomicAdd(out + (int64_t)kStride * p + o, v[o]);
  }
};

// Weight blocks of every chunk: acc12[p][0..B) += (scale / tau_c) w w^T, acc12[p][B..2B) +=
// c0_c w w^T (upper triangle 00 01 02 11 12 22 for IQU), w = (1, cos 2psi, sin 2psi).  The
// chunks are contiguous in sample order; a tile that holds a chunk boundary cuts its runs there
// and looks each run's chunk up.
template <int NC>
struct BinWeights {
  static constexpr int NF = NC == 3 ? 2 : 0, NV = NC == 3 ? 6 : 1, NO = 2 * NV;
  const ChunkDesc* desc;
  int n_chunks;
  const void *cosw, *sinw;
  int half_w;
  const double* c0;
  double scale;
  double* acc12;
  int c_lo, c_hi;          // chunks of the tile's first and last sample
  int64_t base;
  __device__ int chunk_of(int64_t s, int lo, int hi) const {
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (desc[mid].off <= s) lo = mid; else hi = mid - 1;
    }
    return lo;
  }
  __device__ void tile(int64_t first, int64_t last, double* shared) {
    base = first;
    c_lo = chunk_of(first, 0, n_chunks - 1);
    c_hi = c_lo;
    if (c_lo + 1 < n_chunks && desc[c_lo + 1].off <= last) c_hi = chunk_of(last, c_lo, n_chunks - 1);
    if (threadIdx.x == 0) {   // one FP64 division a tile, not one a reduction (2.02 -> 0.65 ms)
      shared[0] = scale / desc[c_lo].tau;
      shared[1] = c0[c_lo];
    }
  }
  __device__ bool cut(int i) const {
    return c_hi != c_lo && desc[chunk_of(base + i, c_lo, c_hi)].off == base + i;
  }
  __device__ float load(int f, int64_t s) const { return load_w(f == 0 ? cosw : sinw, half_w, s); }
  __device__ void add(double* v, const float* f) const {
    if constexpr (NC == 3) {
      const double c = widen(f[0]), w = widen(f[1]);
      v[1] += c;
      v[2] += w;
      v[3] = fma(c, c, v[3]);
      v[4] = fma(c, w, v[4]);
      v[5] = fma(w, w, v[5]);
    }
  }
  __device__ void close(double* v, int len) const { v[0] = (double)len; }
  __device__ void emit(int p, int o, const double* v, int64_t s, const double* shared) const {
    double f = shared[o < NV ? 0 : 1];
    if (c_hi != c_lo) {
      const int c = chunk_of(s, c_lo, c_hi);
      f = o < NV ? scale / desc[c].tau : c0[c];
    }
    atomicAdd(acc12 + (int64_t)NO * p + o, f * v[o < NV ? o : o - NV]);
  }
};

}  // namespace mm
