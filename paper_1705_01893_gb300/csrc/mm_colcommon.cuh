// Device code shared by the column passes of the messenger step and of its adjoint:
// kernel parameters, pointing gathers, the reduce-by-pixel binning of four samples per
// lane, and the first-pass sources / last-pass sink of the column DFTs.
#pragma once

#include "mm_internal.cuh"

namespace mm {

struct ColParams {
  const ChunkDesc* desc;
  const int* chunks;
  Group g;
  // pointing in tile order: the samples of tile (chunk, column block cb) are contiguous,
  // row j1 after row j1 - 1, 2*CB samples per row (see k_tile_pointing)
  const int32_t* __restrict__ pix;
  const void* cosw;
  const void* sinw;
  int half_w;          // weights are FP16
  const void* map4;    // float4 [n_pix] (IQU) or float [n_pix] (T)
  const float* tod;
  float2* ybuf;        // batch slot: chunk ci of the batch at ybuf + ci * M
  int count;           // chunks in the batch
  double* acc;         // planar FP64 accumulators: component k of pixel p at k * acc_stride + p
  int64_t acc_stride;  // n_pix
  // composite pointing (App. B): P = ga P_1 + gb P_2, the second component in tile order too
  const int32_t* __restrict__ pix2;
  const void* cosw2;
  const void* sinw2;
  float ga, gb;
};

// The column kernels' parameters for batch b (plan-owned tile-order pointing, map, buffers).
ColParams make_col_params(const mm_plan_s* p, const Batch& b);

// Four consecutive samples (s a multiple of 4): one 16-byte load per stream.
__device__ __forceinline__ float4 load_w4(const void* w, int half_w, int64_t s) {
  if (half_w) {
    const uint2 b = __ldcs(reinterpret_cast<const uint2*>(static_cast<const __half*>(w) + s));
    const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&b.x));
    const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&b.y));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
  }
  return __ldcs(reinterpret_cast<const float4*>(static_cast<const float*>(w) + s));
}

// (P m) of two consecutive samples; the weights of an excluded one (pixel -1) must be finite, as
// those of the tile-order copies are (included_w).  The two share a pixel more often than not, and
// then one map load serves both: the gathers are short of L1 requests (a vertical sweep touches a
// line per pixel), not of bytes.  256^2, 4 x 2^20: 1523 -> 1461 us per 21 iterations; the 20-step
// gradient 6424 -> 6009 us; 512^2, 8 x 2^22: 435 -> 432 us an iteration.
// kShare: on for IQU.  T-only loads are a quarter of the size, and the second one's wait for the
// compare of the pixels costs more than it saves (forward columns of 250 x 2^14 samples 14.3 us
// against 20.7, 1000 x 2^12 16.5 / 20.8; 4 iterations of 16 x 2^18 220 / 228), but for the long
// columns in narrower tiles (4 iterations of 2 x 2^24 samples 1369 us sharing, 1408 not; 4 x 2^23
// 1316 / 1324).
template <int NC, bool kShare = NC == 3>
__device__ __forceinline__ float2 gather_two(const ColParams& q, int p0, int p1, float c0, float c1,
                                             float s0, float s1) {
  if constexpr (NC == 1) {
    const float* map = reinterpret_cast<const float*>(q.map4);
    const float a = p0 < 0 ? 0.f : __ldg(map + p0);
    float b = a;
    if (!kShare || p1 != p0) b = p1 < 0 ? 0.f : __ldg(map + p1);
    return make_float2(a, b);
  } else {
    const float4* map = reinterpret_cast<const float4*>(q.map4);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (p0 >= 0) a = __ldg(map + p0);
    float4 b = a;
    if (p1 != p0) b = p1 < 0 ? make_float4(0.f, 0.f, 0.f, 0.f) : __ldg(map + p1);
    return make_float2(fmaf(s0, a.z, fmaf(c0, a.y, a.x)), fmaf(s1, b.z, fmaf(c1, b.y, b.x)));
  }
}

// (P m) of four consecutive samples of tile-order pointing; kAnyWeights: of a caller's arrays, whose
// excluded samples may have any weights.
template <int NC, bool kAnyWeights = false>
__device__ __forceinline__ float4 gather4(const ColParams& q, int64_t s) {
  const int4 p = __ldcs(reinterpret_cast<const int4*>(q.pix + s));
  float4 c = make_float4(0.f, 0.f, 0.f, 0.f), w = c;
  if constexpr (NC == 3) {
    c = load_w4(q.cosw, q.half_w, s);
    w = load_w4(q.sinw, q.half_w, s);
    if (kAnyWeights && (p.x | p.y | p.z | p.w) < 0) {   // rarely taken: selects on every sample cost 6%
      if (p.x < 0) c.x = w.x = 0.f;
      if (p.y < 0) c.y = w.y = 0.f;
      if (p.z < 0) c.z = w.z = 0.f;
      if (p.w < 0) c.w = w.w = 0.f;
    }
  }
  const float2 lo = gather_two<NC>(q, p.x, p.y, c.x, c.y, w.x, w.y);
  const float2 hi = gather_two<NC>(q, p.z, p.w, c.z, c.w, w.z, w.w);
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// One FP64 add per component into the planar accumulators.  Planar, because the lanes of a
// warp close runs on neighbouring pixels: one reduction instruction then touches a third of
// the L2 sectors it would with [n_pix][3] (measured on 8 x 2^22 samples: 160 -> 141 us per
// binning launch, which is bound by L2 reduction requests).
template <int NC>
__device__ __forceinline__ void emit_run(double* acc, int64_t stride, int p, float a0, float a1,
                                         float a2, uint64_t pol) {
  if (p < 0) return;
  double* a = acc + p;
  red_add_f64(a, f32_to_f64(a0), pol);
  if constexpr (NC == 3) {
    red_add_f64(a + stride, f32_to_f64(a1), pol);
    red_add_f64(a + 2 * stride, f32_to_f64(a2), pol);
  }
}

// P^T t for samples s..s+3 (t4 = t_s..t_s+3), one lane of a row of ROWL lanes (4 ROWL
// consecutive samples; ROWL = 8, 4 or 2, a power of two dividing the warp).
// Reduce by pixel: runs inside the lane are summed in registers; runs that cross lanes are
// closed by a linear-recurrence scan over the lanes of the row (S_u = X_u + G_u S_{u+1},
// X_u = the lane's leading run when it continues the previous lane's trailing run, G_u = the
// lane is one such run and the next lane continues it).  Each run's first sample's lane
// issues one FP64 add per component.
template <int NC, int ROWL>
__device__ __forceinline__ void bin4(double* acc, int64_t acc_stride, int4 p4, float4 t4, float4 c, float4 w,
                                     int qpos) {
  static_assert(ROWL == 2 || ROWL == 4 || ROWL == 8, "rows of 2, 4 or 8 lanes");
  const uint64_t pol = l2_policy_evict_last();
  const int p[4] = {p4.x, p4.y, p4.z, p4.w};
  const float tv[4] = {t4.x, t4.y, t4.z, t4.w};
  float v[3][4];
  const float cw[4] = {c.x, c.y, c.z, c.w}, sw[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[0][i] = tv[i];
    v[1][i] = tv[i] * cw[i];
    v[2][i] = tv[i] * sw[i];
  }
  const bool b1 = p[1] != p[0], b2 = p[2] != p[1], b3 = p[3] != p[2];
  const int prev3 = __shfl_up_sync(0xffffffffu, p[3], 1);
  const bool cont = qpos != 0 && p[0] == prev3;
  if (__all_sync(0xffffffffu, !b1 && !b3 && !cont)) {
    // every lane holds one pixel, or two of two samples each, and none runs on into the next
    // lane (an even number of samples per pixel): no scan, at most two runs.  4 samples per
    // pixel, 512^2, 8 x 2^22: 432 -> 414 us an iteration; PCG on it 4137 -> 3978 us per 8.
    float h[2][3];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      h[0][k] = v[k][0] + v[k][1];
      h[1][k] = v[k][2] + v[k][3];
      if (!b2) h[0][k] += h[1][k];
    }
    emit_run<NC>(acc, acc_stride, p[0], h[0][0], h[0][1], h[0][2], pol);
    if (b2) emit_run<NC>(acc, acc_stride, p[2], h[1][0], h[1][1], h[1][2], pol);
    return;
  }
  const bool single = !(b1 || b2 || b3);
  const int f = b1 ? 1 : (b2 ? 2 : (b3 ? 3 : 4));   // leading run [0, f)
  const int l = b3 ? 3 : (b2 ? 2 : (b1 ? 1 : 0));   // trailing run [l, 4)
  float lead[3], trail[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    lead[k] = 0.f;
    trail[k] = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      lead[k] += i < f ? v[k][i] : 0.f;
      trail[k] += i >= l ? v[k][i] : 0.f;
    }
  }
  float S[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) S[k] = cont ? lead[k] : 0.f;
  bool Gs = cont && single && qpos != ROWL - 1;
#pragma unroll
  for (int d = 1; d < ROWL; d <<= 1) {
    float Sd[3];
#pragma unroll
    for (int k = 0; k < NC; ++k) Sd[k] = __shfl_down_sync(0xffffffffu, S[k], d);
    const bool Gd = __shfl_down_sync(0xffffffffu, Gs, d);
    if (Gs) {
#pragma unroll
      for (int k = 0; k < NC; ++k) S[k] += Sd[k];
    }
    Gs = Gs && Gd;
  }
  float carry[3];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    const float cd = __shfl_down_sync(0xffffffffu, S[k], 1);
    carry[k] = qpos != ROWL - 1 ? cd : 0.f;
  }
  if (!(single && cont))
    emit_run<NC>(acc, acc_stride, p[3], trail[0] + carry[0], trail[1] + carry[1], trail[2] + carry[2], pol);
  if (!cont && !single) emit_run<NC>(acc, acc_stride, p[0], lead[0], lead[1], lead[2], pol);
  if (b1 && l > 1) {   // middle run [1, e)
    const bool two = b2;
    emit_run<NC>(acc, acc_stride, p[1], two ? v[0][1] : v[0][1] + v[0][2], two ? v[1][1] : v[1][1] + v[1][2],
                 two ? v[2][1] : v[2][1] + v[2][2], pol);
  }
  if (b2 && l > 2) emit_run<NC>(acc, acc_stride, p[2], v[0][2], v[1][2], v[2][2], pol);
}

// g_a P_a^T t + g_b P_b^T t for the same samples (App. B).
template <int NC, int ROWL>
__device__ __forceinline__ void scatter4_pair(const ColParams& q, int64_t s, float4 t4, int qpos) {
#pragma unroll 1
  for (int k = 0; k < 2; ++k) {
    const float g = k ? q.gb : q.ga;
    const int4 p4 = __ldcs(reinterpret_cast<const int4*>((k ? q.pix2 : q.pix) + s));
    float4 c = make_float4(0.f, 0.f, 0.f, 0.f), w = c;
    if constexpr (NC == 3) {
      c = load_w4(k ? q.cosw2 : q.cosw, q.half_w, s);
      w = load_w4(k ? q.sinw2 : q.sinw, q.half_w, s);
    }
    bin4<NC, ROWL>(q.acc, q.acc_stride, p4, make_float4(g * t4.x, g * t4.y, g * t4.z, g * t4.w), c, w, qpos);
  }
}

template <int NC, int ROWL = 8>
__device__ __forceinline__ void scatter4(const ColParams& q, int64_t s, float4 t4, int qpos) {
  const int4 p4 = __ldcs(reinterpret_cast<const int4*>(q.pix + s));
  float4 c = make_float4(0.f, 0.f, 0.f, 0.f), w = c;
  if constexpr (NC == 3) {
    c = load_w4(q.cosw, q.half_w, s);
    w = load_w4(q.sinw, q.half_w, s);
  }
  bin4<NC, ROWL>(q.acc, q.acc_stride, p4, t4, c, w, qpos);
}

// First-pass sources and last-pass sink of the column DFTs.  Element (b, i) of a tile is
// column j2 = j2_0 + b, row j1 = i: samples s = base + 2 (i M2 + b) and s + 1.
template <int NC, int CB>
struct SrcGather {   // z = ((P m)_s, (P m)_s+1), Eq. 1; tile-ordered pointing from `tbase`
  const ColParams* q;
  int64_t tbase;
  __device__ __forceinline__ float2 operator()(int b, int i) const {
    const int64_t s = tbase + 2 * (CB * i + b);
    const int2 p = __ldcs(reinterpret_cast<const int2*>(q->pix + s));
    float cw0 = 0.f, cw1 = 0.f, sw0 = 0.f, sw1 = 0.f;
    if constexpr (NC == 3) {
      if (q->half_w) {
        const float2 c = __half22float2(__ldcs(reinterpret_cast<const __half2*>(static_cast<const __half*>(q->cosw) + s)));
        const float2 w = __half22float2(__ldcs(reinterpret_cast<const __half2*>(static_cast<const __half*>(q->sinw) + s)));
        cw0 = c.x; cw1 = c.y; sw0 = w.x; sw1 = w.y;
      } else {
        const float2 c = __ldcs(reinterpret_cast<const float2*>(static_cast<const float*>(q->cosw) + s));
        const float2 w = __ldcs(reinterpret_cast<const float2*>(static_cast<const float*>(q->sinw) + s));
        cw0 = c.x; cw1 = c.y; sw0 = w.x; sw1 = w.y;
      }
    }
    return gather_two<NC, NC == 3 || (CB < kColCB)>(*q, p.x, p.y, cw0, cw1, sw0, sw1);
  }
};

template <int NC, int CB>
struct SrcGather2 {   // z of g_a P_a m + g_b P_b m (App. B)
  const ColParams* q;
  int64_t tbase;
  __device__ __forceinline__ float2 operator()(int b, int i) const {
    ColParams second{};
    second.pix = q->pix2;
    second.cosw = q->cosw2;
    second.sinw = q->sinw2;
    second.half_w = q->half_w;
    second.map4 = q->map4;
    const float2 u = SrcGather<NC, CB>{q, tbase}(b, i), v = SrcGather<NC, CB>{&second, tbase}(b, i);
    return make_float2(fmaf(q->gb, v.x, q->ga * u.x), fmaf(q->gb, v.y, q->ga * u.y));
  }
};

struct SrcTod {      // z = (d_s, d_s+1)
  const float* tod;
  int64_t base;
  int M2;
  __device__ __forceinline__ float2 operator()(int b, int i) const {
    return __ldcs(reinterpret_cast<const float2*>(tod + base + 2ll * ((int64_t)i * M2 + b)));
  }
};

// The four-step twiddles of column tile cb into shared memory (four_step_n(M1, kColLo) x CB
// entries); ready after the next barrier.
template <int M1, int CB, int T>
__device__ __forceinline__ void load_col_twiddles(float2* s4, const Group& g, int cb) {
  constexpr int N = four_step_n(M1, kColLo) * CB;
  const float2* src = g.tw_c4 + (int64_t)cb * N;
#pragma unroll
  for (int i = threadIdx.x; i < N; i += T) s4[i] = __ldg(src + i);
  // a one-pass column DFT has no barrier of its own before its output
  if constexpr (M1 <= 16) __syncthreads();
}

// y[k1][j2] = Z * w_M^(k1 j2): the four-step twiddle on the way out.  kStream: the
// intermediate is written with evict-first priority (separate pass kernels, whose next
// reader comes a whole batch later), leaving L2 to the map and the accumulators.
template <int M1, int CB, bool kStream = false>
struct DstY {
  float2* y;
  const float2* s4;    // load_col_twiddles
  int j2_0;
  int M2;
  __device__ __forceinline__ void operator()(int b, int k1, float2 v) const {
    float2 w = s4[(k1 & (four_step_lo(M1, kColLo) - 1)) * CB + b];
    if constexpr (M1 > kColLo) w = cmul(s4[(kColLo + k1 / kColLo) * CB + b], w);
    const float2 o = cmul(v, w);
    if constexpr (kStream) __stcs(y + (int64_t)k1 * M2 + j2_0 + b, o);
    else y[(int64_t)k1 * M2 + j2_0 + b] = o;
  }
};

// The same with the plan-wide two-level table, for 32-point columns (see k_col_forward) and the
// transform of the data: that runs once per data set, and its rounding reaches every later iterate
// through d~ (1/f noise spreads it over the high frequencies), so it stays as it was.
struct DstYTable {
  float2* y;
  const Group* g;
  int j2_0;
  int M2;
  __device__ __forceinline__ void operator()(int b, int k1, float2 v) const {
    const int j2 = j2_0 + b;
    __stcs(y + (int64_t)k1 * M2 + j2, cmul(v, tw_big(*g, k1 * j2)));
  }
};

// Filtered spectrum rows for the inverse column DFTs.  kStream: the last read of the
// intermediate (separate pass kernel), evict-first; otherwise L2 only, because in the fused
// iteration kernel other CTAs wrote these rows in this launch.
template <bool kStream = false>
struct SrcY {
  const float2* y;
  int j2_0;
  int M2;
  __device__ __forceinline__ float2 operator()(int b, int k1) const {
    if constexpr (kStream) return __ldcs(y + (int64_t)k1 * M2 + j2_0 + b);
    return __ldcg(y + (int64_t)k1 * M2 + j2_0 + b);
  }
};

}  // namespace mm
