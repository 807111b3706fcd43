// Exact binning of samples into per-pixel FP64 sums for the set-up and the operators (weight
// blocks, P^T of a caller's timestream, the allocation-free binned map): sums over runs of
// consecutive samples on one pixel first, one FP64 reduction per run and sum afterwards.
//
// What bounds it: a reduction per sample and sum saturates the L2's atomic units (12 per
// sample for the weight blocks: 1.90 ms for 8 x 2^22 samples), and FP64 arithmetic runs on a
// pipe of about two lanes per SM and clock.  So a lane takes four consecutive samples and adds
// them up while they stay on one pixel (5 to 8 FP64 instructions a sample, products and sums
// contracted, no lane idle); where a run of the lane ends, its sums go through shared memory and
// are handed out again one (run, sum) per lane, so that a warp's reductions cover the
// consecutive words of two to ten pixels instead of 32 scattered ones.  Lists of whole runs, a
// run a thread, leave the FP64 pipe half idle where the runs differ in length (P^T of 2 M samples
// on a diagonal raster 31 us, 24.7 so).  Measured on 512^2 IQU rasters at 4 samples per pixel:
// weight blocks of 8 x 2^22 samples 1900 -> 566 us, P^T 425 -> 239 us, binned map of 2 x 2^22
// samples 349 -> 150 us.
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

constexpr int kBinWarps = 8, kBinThreads = 32 * kBinWarps;

// Op: NF float streams per sample (load), NV sums per run (add), NO outputs per run (emit).
// Samples [n0, n1); samples with a pixel outside [0, n_pix) are skipped.  Op::tile(first,
// last, shared) prepares per-tile state (every thread, before a barrier); Op::cut(i) marks a tile
// position that starts a run whatever its pixel; Op::kPerSample, Op::one(pixel, s): a single sum
// that may go out sample by sample.
template <class Op>
__global__ void __launch_bounds__(kBinThreads) k_run_bin(Op op, const int32_t* __restrict__ pix,
                                                         int64_t n0, int64_t n1, int64_t n_pix, int segs) {
  constexpr int NF = Op::NF, NV = Op::NV, NO = Op::NO;
  const int tile_n = kBinThreads * 4 * segs;   // samples of a CTA, `segs` rounds of 1024
  constexpr int SV = NV | 1;   // odd stride: the sums of neighbouring runs on different banks
  __shared__ double s_val_[kBinWarps][32 * SV];
  __shared__ int2 s_at_[kBinWarps][32];      // pixel, tile position
  __shared__ double s_op[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* s_val = s_val_[warp];
  int2* s_at = s_at_[warp];
  const int64_t tile = n0 + (int64_t)blockIdx.x * tile_n;
  op.tile(tile, (n1 - tile < tile_n ? n1 : tile + tile_n) - 1, s_op);
  __syncthreads();
  for (int g = 0; g < segs; ++g) {
    const int at = ((g * kBinWarps + warp) * 32 + lane) * 4;   // the lane's first sample in the tile
    if (tile + at - 4 * lane >= n1) break;   // warp-uniform
    // One sum a run and short runs: a reduction per sample, 32 consecutive samples at a time, is
    // the cheaper way (a run's sums of one word gain nothing from being handed out again).  P^T of
    // 8 M T-only samples, by samples per pixel, so / by runs: 1: 26.0 / 47.4 us, 3: 26.1 / 30.9,
    // 4: 26.3 / 29.0, 16: 43.4 / 31.0; hence from 24 runs in 128 samples on (the count makes long
    // runs 2 us slower).
    if constexpr (Op::kPerSample) {
      int q[4], heads = 0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t s = tile + at - 3 * lane + 32 * u;
        q[u] = s < n1 ? pix[s] : -1;
        if (q[u] >= n_pix) q[u] = -1;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int before = __shfl_up_sync(0xffffffffu, q[u], 1);
        heads += __popc(__ballot_sync(0xffffffffu, q[u] >= 0 && (lane == 0 || q[u] != before)));
      }
      if (heads >= 24) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (q[u] >= 0) op.one(q[u], tile + at - 3 * lane + 32 * u);
        continue;
      }
    }
    int p[5];
    float f[4][NF > 0 ? NF : 1];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t s = tile + at + k;
      const bool in = s < n1;
      p[k] = in ? pix[s] : -1;
      if (p[k] >= n_pix) p[k] = -1;
#pragma unroll
      for (int j = 0; j < NF; ++j) f[k][j] = in ? op.load(j, s) : 0.f;
    }
    p[4] = -2;
    double v[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] = 0.0;
    int len = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool on = p[k] >= 0;
      if (on) {
        op.add(v, f[k]);
        ++len;
      }
      // runs that end at this sample
      const bool end = on && (p[k + 1] != p[k] || (k < 3 && op.cut(at + k + 1)));
      const unsigned m = __ballot_sync(0xffffffffu, end);
      if (m == 0) continue;
      if (end) {
        const int r = __popc(m & ((1u << lane) - 1u));
        op.close(v, len);
        s_at[r] = make_int2(p[k], at + k);
#pragma unroll
        for (int j = 0; j < NV; ++j) {
          s_val[r * SV + j] = v[j];
          v[j] = 0.0;
        }
        len = 0;
      }
      __syncwarp();
      const int nr = __popc(m);
      for (int t = lane; t < nr * NO; t += 32) {
        const int r = t / NO, o = t - r * NO;
        const int2 e = s_at[r];
        op.emit(e.x, o, s_val + r * SV, tile + e.y, s_op);
      }
      __syncwarp();
    }
  }
}

template <class Op>
static cudaError_t launch_run_bin(const Op& op, const int32_t* pix, int64_t n0, int64_t n1,
                                  int64_t n_pix, cudaStream_t st) {
  if (n1 <= n0) return cudaSuccess;
  // four rounds a CTA where that still gives every SM several CTAs
  const int segs = n1 - n0 < (1 << 22) ? 1 : 4, tile = kBinThreads * 4 * segs;
  k_run_bin<Op><<<(unsigned)((n1 - n0 + tile - 1) / tile), kBinThreads, 0, st>>>(op, pix, n0, n1, n_pix, segs);
  return cudaGetLastError();
}

// P^T t into interleaved [n_pix][NC] sums.
template <int NC>
struct BinPT {
  static constexpr int NF = NC == 3 ? 3 : 1, NV = NC, NO = NC;
  static constexpr bool kPerSample = NC == 1;
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
  __device__ void one(int p, int64_t s) const { atomicAdd(out + p, widen(tod[s])); }   // NC = 1
};

// Normal-equation sums of the unit-weight binned map, kStride doubles per pixel: hits, then
// (IQU) c, s, cc, cs, ss, d, dc, ds or (T) d.
template <int NC, int kStride>
struct BinNormal {
  static constexpr int NF = NC == 3 ? 3 : 1, NV = NC == 3 ? 9 : 2, NO = NV;
  static constexpr bool kPerSample = false;
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
  static constexpr bool kPerSample = false;
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
