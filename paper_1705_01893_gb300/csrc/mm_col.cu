// Column passes of the four-step FFT, fused with the pointing operators:
//   kernel A (k_col_forward): gather (P m)_s (Eq. 1) or read d_s, pack z_j = x_2j + i x_2j+1,
//            length-M1 column DFTs, twiddle w_M^{k1 j2}, write the row-layout intermediate;
//   kernel C (k_col_inverse): length-M1 inverse column DFTs of the filtered spectrum, unpack
//            t_s, and bin P^T t into FP64 per-pixel accumulators (the co-addition of t in
//            the map step of Sec. 2.1).
// Each CTA owns CB consecutive columns j2 of one chunk, i.e. runs of 2*CB consecutive
// samples at M1 places, so every global access is a contiguous run.
#include "mm_colcommon.cuh"

namespace mm {

// Persistent over the batch's tiles (chunk ci, column block cb).
template <int M1, int CB, int T, int NC, int SRC, bool ROOMY>
__global__ void __launch_bounds__(T, pass_ctas(T, 8, ROOMY)) k_col_forward(ColParams q) {
  extern __shared__ float2 sm[];
  // the tile's four-step twiddles from shared memory, but for 32-point columns, which use each
  // entry once (4 T-only iterations of 1000 x 2^12 samples 266 us without, 276 with; 16 points, whose
  // one pass hides the copy, 4000 x 2^10: 328 / 311; longer columns use entries many times)
  constexpr bool kStage = SRC != kSrcTod && M1 != 32;
  __shared__ float2 s4[kStage ? four_step_n(M1, kColLo) * CB : 1];
  const int M2 = q.g.M2;
  const int tpc = M2 / CB;
  const int ntiles = q.count * tpc;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int ci = t / tpc;
    const ChunkDesc d = q.desc[q.chunks[ci]];
    const int cb = t % tpc;
    const int j2_0 = cb * CB;
    if constexpr (SRC == kSrcTod) {
      smem_fft<M1, CB, ColLayout<CB>, T, -1>(sm, q.g.tw_col, SrcTod{q.tod, d.off + 2ll * j2_0, M2},
                                             DstYTable{q.ybuf + (int64_t)ci * d.M, &q.g, j2_0, M2});
    } else {
      using Src = typename std::conditional<SRC == kSrcGather2, SrcGather2<NC, CB>, SrcGather<NC, CB>>::type;
      const Src src{&q, d.off + (int64_t)cb * (2 * CB * M1)};
      if constexpr (kStage) {
        load_col_twiddles<M1, CB, T>(s4, q.g, cb);
        smem_fft<M1, CB, ColLayout<CB>, T, -1>(sm, q.g.tw_col, src,
                                               DstY<M1, CB, true>{q.ybuf + (int64_t)ci * d.M, s4, j2_0, M2});
      } else {
        smem_fft<M1, CB, ColLayout<CB>, T, -1>(sm, q.g.tw_col, src,
                                               DstYTable{q.ybuf + (int64_t)ci * d.M, &q.g, j2_0, M2});
      }
    }
    __syncthreads();
  }
}

template <int M1, int CB, int T, int NC, bool COMP, bool ROOMY>
__global__ void __launch_bounds__(T, pass_ctas(T, 8, ROOMY)) k_col_inverse(ColParams q) {
  extern __shared__ float2 sm[];
  const int M2 = q.g.M2;
  const int tpc = M2 / CB;
  const int ntiles = q.count * tpc;
  constexpr int RUN = 2 * CB;
  constexpr int NS = M1 * RUN;
  constexpr int ROWL = RUN / 4;   // lanes per row of the tile (4 samples per lane)
  static_assert((RUN == 32 || RUN == 16 || RUN == 8) && (NS / 4) % T == 0 && T % 32 == 0,
                "rows of 8, 4 or 2 lanes and a warp-uniform scatter loop");
  using Lay = ColLayout<CB>;
  const float* smf = reinterpret_cast<const float*>(sm);
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int ci = t / tpc;
    const ChunkDesc d = q.desc[q.chunks[ci]];
    const int cb = t % tpc;
    smem_fft<M1, CB, ColLayout<CB>, T, +1>(sm, q.g.tw_col,
                                           SrcY<true>{q.ybuf + (int64_t)ci * d.M, cb * CB, M2});
    // tile-ordered pointing: the tile's samples are contiguous, in the same order as t
    const int64_t tbase = d.off + (int64_t)cb * NS;
#pragma unroll 4
    for (int e4 = threadIdx.x; e4 < NS / 4; e4 += T) {
      const int e = 4 * e4;
      // sample e = 2 (i CB + b) + h sits at float 2 Lay::at(b, i) + h; a lane's 4 samples
      // lie in one row i
      const int i = e / RUN;
      const int so = e + (Lay::kPad ? 2 * (i >> 4) * Lay::kPad : 0);
      const float4 t4 = *reinterpret_cast<const float4*>(smf + so);
      if constexpr (COMP) scatter4_pair<NC, ROWL>(q, tbase + e, t4, e4 & (ROWL - 1));
      else scatter4<NC, ROWL>(q, tbase + e, t4, e4 & (ROWL - 1));
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------ launchers


// Copy the caller's pointing into tile order: sample 2 (j1 M2 + j2) + h of a chunk goes to
// cb (2 CB M1) + j1 (2 CB) + 2 (j2 - cb CB) + h with cb = j2 / CB (CB = col_cb(M1), the
// column kernels' tile width).  A tile's rows are runs of 2 CB >= 8 samples on both sides, so
// four samples move at once, 16 bytes (8 for FP16 weights); all sizes are powers of two, so
// the indices are shifts.  Reads the caller's arrays element by element when they don't start
// on such a boundary.  8 x 2^22 samples with FP32 weights: 250 -> 135 us (one sample a thread
// with 64-bit divisions before).  Excluded samples (pixel -1), which may have any weights (NaN,
// inf), get weight 0, so that the gathers need not select on the pixel: that select on every
// sample and iteration made 512^2, 8 x 2^22 4% slower, 2048^2, 32 x 2^24 3% and PCG 7%.
template <typename V4, typename V>
__device__ __forceinline__ V4 load4(const void* p, int64_t i, bool aligned) {
  if (aligned) return *reinterpret_cast<const V4*>(static_cast<const V*>(p) + i);
  V4 r;
  V* e = reinterpret_cast<V*>(&r);
#pragma unroll
  for (int k = 0; k < 4; ++k) e[k] = static_cast<const V*>(p)[i + k];
  return r;
}

// Four weights, 0 for excluded samples.
template <typename V4, typename V>
__device__ __forceinline__ V4 included_w(const void* w, int64_t i, bool aligned, int4 p) {
  V4 r = load4<V4, V>(w, i, aligned);
  V* e = reinterpret_cast<V*>(&r);
  if (p.x < 0) e[0] = V(0);
  if (p.y < 0) e[1] = V(0);
  if (p.z < 0) e[2] = V(0);
  if (p.w < 0) e[3] = V(0);
  return r;
}

__global__ void k_tile_pointing(const int32_t* __restrict__ pix, const void* cosw, const void* sinw,
                                int wbytes, int64_t off, int log_m1, int log_m2, int log_row,
                                int aligned, int32_t* __restrict__ tpix, void* tcos, void* tsin) {
  const int o = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (o >= 2 << (log_m1 + log_m2)) return;
  const int w = o & ((1 << log_row) - 1);
  const int j1 = (o >> log_row) & ((1 << log_m1) - 1), cb = o >> (log_row + log_m1);
  const int64_t src = off + (((int64_t)j1 << (log_m2 + 1)) + (cb << log_row) + w), dst = off + o;
  const int4 p = load4<int4, int>(pix, src, aligned & 1);
  *reinterpret_cast<int4*>(tpix + dst) = p;
  if (cosw) {
    if (wbytes == 2) {
      *reinterpret_cast<uint2*>(static_cast<__half*>(tcos) + dst) = included_w<uint2, uint16_t>(cosw, src, aligned & 2, p);
      *reinterpret_cast<uint2*>(static_cast<__half*>(tsin) + dst) = included_w<uint2, uint16_t>(sinw, src, aligned & 2, p);
    } else {
      *reinterpret_cast<float4*>(static_cast<float*>(tcos) + dst) = included_w<float4, float>(cosw, src, aligned & 2, p);
      *reinterpret_cast<float4*>(static_cast<float*>(tsin) + dst) = included_w<float4, float>(sinw, src, aligned & 2, p);
    }
  }
}

cudaError_t launch_tile_pointing(const mm_plan_s* p, cudaStream_t st) {
  const int wb = p->wdtype == MM_W_F16 ? 2 : 4;
  // chunks of the compile-time path start on multiples of 4 samples
  const uintptr_t wm = wb == 2 ? 7 : 15;
  const int aligned = (((uintptr_t)p->pix & 15) == 0 ? 1 : 0) |
                      ((((uintptr_t)p->cosw | (uintptr_t)p->sinw) & wm) == 0 ? 2 : 0);
  const int aligned_b = (((uintptr_t)p->pix_b & 15) == 0 ? 1 : 0) |
                        ((((uintptr_t)p->cos_b | (uintptr_t)p->sin_b) & wm) == 0 ? 2 : 0);
  for (int c = 0; c < p->n_chunks; ++c) {
    const ChunkDesc& d = p->h_desc[c];
    if (p->groups[d.grp].general) continue;   // the general path has its own tile copy
    const unsigned grid = (unsigned)((d.n / 4 + 255) / 256);
    k_tile_pointing<<<grid, 256, 0, st>>>(
        p->pix, p->cosw, p->sinw, wb, d.off, ilog2(d.M1), ilog2(d.M2), ilog2(2 * col_cb(d.M1)), aligned,
        p->tpix, p->tcos, p->tsin);
    if (p->composite)
      k_tile_pointing<<<grid, 256, 0, st>>>(
          p->pix_b, p->cos_b, p->sin_b, wb, d.off, ilog2(d.M1), ilog2(d.M2), ilog2(2 * col_cb(d.M1)), aligned_b,
          p->tpix2, p->tcos2, p->tsin2);
  }
  return cudaGetLastError();
}

static ColParams make_params(const mm_plan_s* p, const Batch& b, const float* tod,
                             const void* map4 = nullptr, float2* ybuf = nullptr) {
  ColParams q;
  const Group& g = p->groups[b.group];
  q.desc = p->d_desc;
  q.chunks = g.chunks + b.first;
  q.count = b.count;
  q.g = g;
  q.pix = p->tpix;
  q.cosw = p->tcos;
  q.sinw = p->tsin;
  q.half_w = p->wdtype == MM_W_F16;
  q.map4 = map4 ? map4 : p->map4;
  q.tod = tod;
  q.ybuf = ybuf ? ybuf : p->ybuf;
  q.acc = p->acc;
  q.pix2 = p->tpix2;
  q.cosw2 = p->tcos2;
  q.sinw2 = p->tsin2;
  q.ga = p->gain_a;
  q.gb = p->gain_b;
  q.acc_stride = acc_stride_of(p->n_pix, p->ncomp);
  return q;
}

ColParams make_col_params(const mm_plan_s* p, const Batch& b) {
  return make_params(p, b, nullptr);
}

template <int M1>
static cudaError_t col_forward_m1(const mm_plan_s* p, const Batch& b, int src, const float* tod,
                                  const void* map4, float2* ybuf, cudaStream_t st) {
  constexpr int kColT = col_threads(M1);
  constexpr int CB = col_cb(M1);
  const ColParams q = make_params(p, b, tod, map4, ybuf);
  const int ntiles = (q.g.M2 / CB) * b.count;
  const size_t smem = sizeof(float2) * ColLayout<CB>::size(M1);
  cudaError_t e;
  int grid = 0;
  const bool iqu = p->ncomp == 3;
  auto pick = [&](auto roomy_) {
    constexpr bool R = decltype(roomy_)::value && kColT != 512;
    return src == kSrcTod ? k_col_forward<M1, CB, kColT, 1, kSrcTod, R>
           : p->composite ? (iqu ? k_col_forward<M1, CB, kColT, 3, kSrcGather2, R> : k_col_forward<M1, CB, kColT, 1, kSrcGather2, R>)
                          : (iqu ? k_col_forward<M1, CB, kColT, 3, kSrcGather, R> : k_col_forward<M1, CB, kColT, 1, kSrcGather, R>);
  };
  auto k = pick(std::false_type{});
  if ((e = pass_grid(pick(std::true_type{}), k, kColT, smem, ntiles, &k, &grid)) != cudaSuccess) return e;
  k<<<grid, kColT, smem, st>>>(q);
  return cudaGetLastError();
}

template <int M1>
static cudaError_t col_inverse_m1(const mm_plan_s* p, const Batch& b, cudaStream_t st) {
  constexpr int kColT = col_threads(M1);
  constexpr int CB = col_cb(M1);
  const ColParams q = make_params(p, b, nullptr);
  const int ntiles = (q.g.M2 / CB) * b.count;
  const size_t smem = sizeof(float2) * ColLayout<CB>::size(M1);
  cudaError_t e;
  int grid = 0;
  const bool iqu = p->ncomp == 3;
  auto pick = [&](auto roomy_) {
    constexpr bool R = decltype(roomy_)::value && kColT != 512;
    return p->composite ? (iqu ? k_col_inverse<M1, CB, kColT, 3, true, R> : k_col_inverse<M1, CB, kColT, 1, true, R>)
                        : (iqu ? k_col_inverse<M1, CB, kColT, 3, false, R> : k_col_inverse<M1, CB, kColT, 1, false, R>);
  };
  auto k = pick(std::false_type{});
  if ((e = pass_grid(pick(std::true_type{}), k, kColT, smem, ntiles, &k, &grid)) != cudaSuccess) return e;
  k<<<grid, kColT, smem, st>>>(q);
  return cudaGetLastError();
}

cudaError_t launch_col_forward(const mm_plan_s* p, const Batch& b, int src, const float* tod,
                               cudaStream_t st) {
  return launch_col_forward_ex(p, b, src, tod, nullptr, nullptr, st);
}

cudaError_t launch_col_forward_ex(const mm_plan_s* p, const Batch& b, int src, const float* tod,
                                  const void* map4, float2* ybuf, cudaStream_t st) {
  if (b.group < 0) {
    if (map4 || ybuf) return cudaErrorInvalidValue;
    return launch_gen_col_forward(p, b, src, tod, st);
  }
  const Group& g = p->groups[b.group];
  switch (g.M1) {
    case 16: return col_forward_m1<16>(p, b, src, tod, map4, ybuf, st);
    case 32: return col_forward_m1<32>(p, b, src, tod, map4, ybuf, st);
    case 64: return col_forward_m1<64>(p, b, src, tod, map4, ybuf, st);
    case 128: return col_forward_m1<128>(p, b, src, tod, map4, ybuf, st);
    case 256: return col_forward_m1<256>(p, b, src, tod, map4, ybuf, st);
    case 512: return col_forward_m1<512>(p, b, src, tod, map4, ybuf, st);
    case 1024: return col_forward_m1<1024>(p, b, src, tod, map4, ybuf, st);
    case 2048: return col_forward_m1<2048>(p, b, src, tod, map4, ybuf, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_col_inverse(const mm_plan_s* p, const Batch& b, cudaStream_t st) {
  if (b.group < 0) return launch_gen_col_inverse(p, b, st);
  const Group& g = p->groups[b.group];
  switch (g.M1) {
    case 16: return col_inverse_m1<16>(p, b, st);
    case 32: return col_inverse_m1<32>(p, b, st);
    case 64: return col_inverse_m1<64>(p, b, st);
    case 128: return col_inverse_m1<128>(p, b, st);
    case 256: return col_inverse_m1<256>(p, b, st);
    case 512: return col_inverse_m1<512>(p, b, st);
    case 1024: return col_inverse_m1<1024>(p, b, st);
    case 2048: return col_inverse_m1<2048>(p, b, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace mm
