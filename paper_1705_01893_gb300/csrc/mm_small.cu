// Messenger iterations of a small plan in one launch.
//
// A plan of a few short chunks spends its iterations on latency: three FFT kernels and the map
// step, each a few CTAs for a few microseconds, one after the other (20.8 us an iteration for one
// chunk of 2^15 samples, 40 us for 12 ragged ones).  Here a thread-block cluster owns a chunk:
// its CTAs split the columns of the four-step FFT, exchange the intermediate through
// distributed shared memory, split the row pairs, filter, and send the rows back, so that
// nothing of the chunk leaves the chip between gather and binning.  The map step is shared out
// over all CTAs between two grid barriers (one cluster: the cluster's own barrier), and one
// launch runs the whole schedule.  What bounds an iteration is then the chain of barriers,
// exchanges and L2 round trips.  Measured: one chunk of 2^15 samples, T-only, 101 iterations
// 2.10 -> 1.16 ms; 12 ragged IQU chunks of 1500 to 12000 samples, 21 iterations 844 -> 321 us.
//
// Lengths are general (radices 2, 3, 4, 5, 8, 16 at run time), with the layouts and scales of
// the other paths: row layout of d~ and Nbar, sums scaled by 1 / (n tau).
#include <cooperative_groups.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "mm_colcommon.cuh"

namespace cg = cooperative_groups;

namespace mm {

constexpr int kSmallThreads = 512;
constexpr int kSmallLambdas = 128;   // iterations per launch (their lambdas travel as arguments)

struct SmallParams {
  const GenChunk* rec;        // [n_chunks]
  const ChunkDesc* desc;      // tau of the noise model in force
  int n_chunks;
  int tile, tables;           // words (float2) of each of the three work buffers, of the kept tables
  const int32_t* __restrict__ pix;
  const void* cosw;
  const void* sinw;
  int half_w;
  const float2* __restrict__ dtab;
  const float* __restrict__ nbar;
  const float* __restrict__ nyq;
  const double* __restrict__ W;
  double* acc;
  void* map4;
  double* map_out;            // written by the last iteration, or nullptr
  double* chi2;               // [n_iter] or nullptr
  int64_t n_pix;
  unsigned* bar;              // grid barrier arrivals, zero at launch
  int* fault;
  int n_polls, n_iter;
  double lambda[kSmallLambdas];
};

// k / d for 0 <= k < 2^22: the approximate reciprocal's quotient is within one of the true one.
struct SmallDiv {
  int d;
  float inv;
  __device__ __forceinline__ explicit SmallDiv(int dd) : d(dd) {
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"((float)dd));
  }
  __device__ __forceinline__ int div(int k) const {
    int q = __float2int_rz((float)k * inv);
    const int r = k - q * d;
    q -= r < 0;
    q += r >= d;
    return q;
  }
};

// A table entry: shared memory when the chunk's tables are kept there, else the read-only path.
template <bool kCache>
__device__ __forceinline__ float2 small_ld(const float2* p) {
  if constexpr (kCache) return *p;
  return __ldg(p);
}

__device__ __forceinline__ int small_lay(int e) { return e + (e >> 4); }

// One Stockham pass of radix R over nq sequences of length L.  Columns (kRows false): element i
// of sequence q at i nq + q; rows: at small_lay(q L + i), one spare word after every 16.
template <int R, int DIR, bool kRows, bool kCache>
__device__ __forceinline__ void small_pass(const float2* src, float2* dst, int L, int Ns, int nq,
                                           const float2* tw) {
  const int nb = SmallDiv(R).div(L), total = nb * nq;
  const SmallDiv dm(kRows ? nb : nq), ds(Ns);
  for (int b = threadIdx.x; b < total; b += kSmallThreads) {
    const int hi = dm.div(b), lo = b - hi * dm.d;
    const int i = kRows ? lo : hi, q = kRows ? hi : lo;
    const int k = i - ds.div(i) * Ns;
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r)
      v[r] = src[kRows ? small_lay(q * L + i + r * nb) : (i + r * nb) * nq + q];
    if (Ns > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) {
        const float2 w = small_ld<kCache>(tw + r * Ns + k);
        v[r] = DIR < 0 ? cmul(v[r], w) : cmulc(v[r], w);
      }
    }
    dftR<R, DIR>(v);
    const int o = (i - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[kRows ? small_lay(q * L + o + r * Ns) : (o + r * Ns) * nq + q] = v[r];
  }
}

// All passes, ping-pong between a and b; returns the buffer that holds the result.
template <int DIR, bool kRows, bool kCache>
__device__ float2* small_dft(float2* a, float2* b, int L, int nr, const int8_t* rad, const float2* tw,
                             int nq) {
  int Ns = 1;
  for (int p = 0; p < nr; ++p) {
    const int R = rad[p];
    switch (R) {
      case 2: small_pass<2, DIR, kRows, kCache>(a, b, L, Ns, nq, tw); break;
      case 3: small_pass<3, DIR, kRows, kCache>(a, b, L, Ns, nq, tw); break;
      case 4: small_pass<4, DIR, kRows, kCache>(a, b, L, Ns, nq, tw); break;
      case 5: small_pass<5, DIR, kRows, kCache>(a, b, L, Ns, nq, tw); break;
      case 8: small_pass<8, DIR, kRows, kCache>(a, b, L, Ns, nq, tw); break;
      default: small_pass<16, DIR, kRows, kCache>(a, b, L, Ns, nq, tw); break;
    }
    __syncthreads();
    float2* t = a; a = b; b = t;
    tw += Ns * R;
    Ns *= R;
  }
  return a;
}

// Every CTA of the grid has arrived `round` times (1, 2, ...).  Bounded like every wait here: on
// expiry, or once any wait has expired, it returns at once with the fault flag set.
__device__ __forceinline__ void small_grid_barrier(const SmallParams& q, unsigned round, int* s_dead) {
  __syncthreads();
  if (threadIdx.x == 0 && !*s_dead) {
    __threadfence();
    atomicAdd(q.bar, 1u);
    const unsigned target = round * gridDim.x;
    for (int n = 0;; ++n) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(q.bar) : "memory");
      if (v >= target) break;
      if (n >= q.n_polls) {
        atomicExch(q.fault, 1);
        *s_dead = 1;
        break;
      }
      if (n > 32) __nanosleep(64);
    }
    __threadfence();
  }
  __syncthreads();
}

// What a CTA keeps of the chunk it works on: the record with its tables (in shared memory when
// kCache), and the constants that cost FP64 instructions or divisions.
struct SmallState {
  GenChunk g;
  float tau, sc, inv_n, lt;   // lt: lambda tau of the iteration
  double inv_nd, tau_d;
  int dead;
};

// kCache: a cluster has one chunk, whose pointing, spectra and tables stay in shared memory over
// all iterations (the fences of the barriers empty L1, so that anything read through it costs an
// L2 round trip each time; the chunk of 2^15 samples takes 18.8 us an iteration with
// the tables in global memory and FP64 divisions in the chain, 11 us without).
template <int NC, bool kCache>
__global__ void __launch_bounds__(kSmallThreads, 1) k_small(SmallParams q) {
  extern __shared__ float2 sm[];
  __shared__ float red[32];
  __shared__ SmallState st;
  cg::cluster_group cl = cg::this_cluster();
  const int S = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int n_cl = gridDim.x / S, my_cl = blockIdx.x / S;
  float2* A = sm;
  float2* B = sm + q.tile;
  float2* X = sm + 2 * q.tile;
  // kCache: d~ of the CTA's rows, the tables, Nbar, pixels and weights of its columns (indexed
  // like the tile, sample h of element e at 2 e + h)
  float2* c_d = sm + 3 * q.tile;
  float2* c_tw = c_d + q.tile;
  float* c_n = reinterpret_cast<float*>(c_tw + q.tables);
  int* c_pix = reinterpret_cast<int*>(c_n + q.tile);
  float* c_cos = reinterpret_cast<float*>(c_pix + 2 * q.tile);
  float* c_sin = c_cos + 2 * q.tile;
  unsigned rounds = 0;
  auto sync_all = [&]() {
    if (n_cl == 1) {
      __threadfence();
      cl.sync();
    } else {
      small_grid_barrier(q, ++rounds, &st.dead);
    }
  };
  auto weight = [&](const void* w, int64_t s) {
    return q.half_w ? __half2float(static_cast<const __half*>(w)[s]) : __ldg(static_cast<const float*>(w) + s);
  };
  if (threadIdx.x == 0) st.dead = 0;
  // A peer's shared memory may be written only between two cluster barriers: one that shows that
  // the peer runs (this one, before the first exchange) and the one at the end, before which none
  // leaves.  A cluster's CTAs are scheduled together, but need not have started together.
  cl.sync();

  for (int it = 0; it < q.n_iter; ++it) {
    const bool lam_inf = isinf(q.lambda[it]);
    for (int ci = my_cl; ci < q.n_chunks; ci += n_cl) {
      const bool fill = !kCache || it == 0;
      if (fill) {
        const int* src = reinterpret_cast<const int*>(q.rec + ci);
        int* dst = reinterpret_cast<int*>(&st.g);
        for (int i = threadIdx.x; i < (int)(sizeof(GenChunk) / 4); i += kSmallThreads) dst[i] = src[i];
        __syncthreads();
      }
      const int M1 = st.g.d.M1, M2 = st.g.d.M2, M = st.g.d.M;
      const bool cplx = st.g.d.cplx != 0;
      const int64_t off = st.g.d.off, spec = st.g.d.spec;
      const int cw = SmallDiv(S).div(M2 + S - 1);            // columns per CTA
      const int j0 = rank * cw, width = max(0, min(cw, M2 - j0));
      const int units = M1 / 2 + 1, upc = SmallDiv(S).div(units + S - 1);   // row units (k1, M1 - k1) per CTA
      const int u0 = rank * upc, nu = max(0, min(upc, units - u0));
      const int nh = cplx ? 1 : 2, lo_mask = (1 << st.g.log_lo) - 1, log_lo = st.g.log_lo;
      const SmallDiv dcw(width > 0 ? width : 1), dm2(M2), dupc(upc), dcwf(cw);
      auto row_of = [&](int sq) { const int u = u0 + (sq >> 1); return (sq & 1) ? M1 - u : u; };
      // tables: per-pass ones of the columns and rows (fewer than 2 L words each), four-step, packing
      const float2* t_col = kCache ? c_tw : st.g.tw_col;
      const float2* t_row = kCache ? c_tw + 2 * M1 : st.g.tw_row;
      const float2* t_lo = kCache ? c_tw + 2 * (M1 + M2) : st.g.tw_lo;
      const float2* t_hi = kCache ? c_tw + 2 * (M1 + M2) + lo_mask + 1 : st.g.tw_hi;
      const float2* t_pa = kCache ? c_tw + 2 * (M1 + M2) + lo_mask + 2 + (M >> log_lo) : st.g.pack_a;
      const float2* t_pb = kCache ? c_tw + 2 * (M1 + M2) + lo_mask + 2 + (M >> log_lo) + M1 : st.g.pack_b;
      if (threadIdx.x == 0) {
        if (fill) {
          const double tau_d = q.desc[st.g.c].tau;
          st.tau_d = tau_d;
          st.tau = (float)tau_d;
          st.inv_n = 1.0f / (float)st.g.d.n;
          st.sc = st.inv_n / st.tau;
          st.inv_nd = 1.0 / (double)st.g.d.n;
        }
        st.lt = lam_inf ? 0.f : (float)(q.lambda[it] * st.tau_d);
      }
      if (kCache && fill) {
        for (int e = threadIdx.x; e < M1 * width; e += kSmallThreads) {
          const int j1 = dcw.div(e), c = e - j1 * width;
          for (int h = 0; h < nh; ++h) {
            const int64_t s = off + ((int64_t)j1 * M2 + j0 + c) * nh + h;
            c_pix[2 * e + h] = q.pix[s];
            if constexpr (NC == 3) {
              c_cos[2 * e + h] = weight(q.cosw, s);
              c_sin[2 * e + h] = weight(q.sinw, s);
            }
          }
        }
        for (int e = threadIdx.x; e < 2 * nu * M2; e += kSmallThreads) {
          const int sq = dm2.div(e), p = e - sq * M2, r = row_of(sq);
          if (r < M1) {
            c_d[e] = q.dtab[spec + (int64_t)r * M2 + p];
            c_n[e] = q.nbar[spec + (int64_t)r * M2 + p];
          }
        }
        auto copy = [&](const float2* dst, const float2* src, int cnt) {
          for (int i = threadIdx.x; i < cnt; i += kSmallThreads) const_cast<float2*>(dst)[i] = src[i];
        };
        int nc = 0, nr = 0;   // words of the pass tables
        for (int p = 0, ns = 1; p < st.g.nr1; ++p) { nc += ns * st.g.rad1[p]; ns *= st.g.rad1[p]; }
        for (int p = 0, ns = 1; p < st.g.nr2; ++p) { nr += ns * st.g.rad2[p]; ns *= st.g.rad2[p]; }
        copy(t_col, st.g.tw_col, nc);
        copy(t_row, st.g.tw_row, nr);
        copy(t_lo, st.g.tw_lo, lo_mask + 1);
        copy(t_hi, st.g.tw_hi, ((M - 1) >> log_lo) + 1);
        copy(t_pa, st.g.pack_a, M1);
        copy(t_pb, st.g.pack_b, M2);
        // the pointing is read back by the thread that wrote it, the rest after later barriers
      }
      auto big = [&](int e) { return cmul(small_ld<kCache>(t_hi + (e >> log_lo)), small_ld<kCache>(t_lo + (e & lo_mask))); };
      // ---- gather (P m), packed z = x_2j + i x_2j+1 (odd n: x_j)
      for (int e0 = threadIdx.x; e0 < M1 * width; e0 += 4 * kSmallThreads) {
        int px[4][2];
        float cs[4][2], sn[4][2];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int e = e0 + u * kSmallThreads;
          const bool on = e < M1 * width;
          int64_t s = 0;
          if constexpr (!kCache) {
            const int j1 = on ? dcw.div(e) : 0, c = e - j1 * width;
            s = off + ((int64_t)j1 * M2 + j0 + c) * nh;
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            px[u][h] = -1;
            cs[u][h] = sn[u][h] = 0.f;
            if (on && h < nh) {
              if constexpr (kCache) {
                px[u][h] = c_pix[2 * e + h];
                if constexpr (NC == 3) { cs[u][h] = c_cos[2 * e + h]; sn[u][h] = c_sin[2 * e + h]; }
              } else {
                px[u][h] = __ldg(q.pix + s + h);
                if constexpr (NC == 3) { cs[u][h] = weight(q.cosw, s + h); sn[u][h] = weight(q.sinw, s + h); }
              }
            }
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int e = e0 + u * kSmallThreads;
          float z[2] = {0.f, 0.f};
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            // plain loads: the map was written in this launch (ordered by the grid barrier)
            if (px[u][h] < 0) continue;
            if constexpr (NC == 1) {
              z[h] = reinterpret_cast<const float*>(q.map4)[px[u][h]];
            } else {
              const float4 m = reinterpret_cast<const float4*>(q.map4)[px[u][h]];
              z[h] = fmaf(sn[u][h], m.z, fmaf(cs[u][h], m.y, m.x));
            }
          }
          if (e < M1 * width) A[e] = make_float2(z[0], z[1]);
        }
      }
      __syncthreads();
      // ---- column DFTs, twiddle, rows to their owners
      if (width > 0) {
        const float2* r = small_dft<-1, false, kCache>(A, B, M1, st.g.nr1, st.g.rad1, t_col, width);
        for (int e = threadIdx.x; e < M1 * width; e += kSmallThreads) {
          const int k1 = dcw.div(e), j2 = j0 + e - k1 * width;
          const float2 v = cmul(r[e], big(k1 * j2));
          const int kc = k1 == 0 ? 0 : M1 - k1;
          const int u = k1 <= kc ? k1 : kc, own = dupc.div(u);
          const int sq = 2 * (u - own * upc) + (k1 > kc && k1 != 0 ? 1 : 0);
          *cl.map_shared_rank(X + small_lay(sq * M2 + j2), own) = v;
        }
      }
      cl.sync();
      // ---- row DFTs, split, filter, chi^2, merge, inverse row DFTs (as in the other row jobs)
      float x2 = 0.f;
      if (nu > 0) {
        float2* z = small_dft<-1, true, kCache>(X, A, M2, st.g.nr2, st.g.rad2, t_row, 2 * nu);
        const float tau = st.tau, sc = st.sc, lt = st.lt;
        auto filt = [&](float2 Xv, float2 D, float nbv) -> float2 {
          if (lam_inf) return cscale(D, sc);
          const float r = __fdividef(sc, lt + nbv);
          return make_float2((lt * D.x + nbv * Xv.x) * r, (lt * D.y + nbv * Xv.y) * r);
        };
        auto dval = [&](int sq, int r, int p) { return kCache ? c_d[sq * M2 + p] : __ldg(q.dtab + spec + (int64_t)r * M2 + p); };
        auto nval = [&](int sq, int r, int p) { return kCache ? c_n[sq * M2 + p] : __ldg(q.nbar + spec + (int64_t)r * M2 + p); };
        if (cplx) {
          for (int e = threadIdx.x; e < 2 * nu * M2; e += kSmallThreads) {
            const int sq = dm2.div(e), p = e - sq * M2, r = row_of(sq);
            if ((sq & 1) && u0 + (sq >> 1) == 0) continue;   // row 0 pairs with itself (odd M1)
            const float2 Xv = z[small_lay(e)], D = dval(sq, r, p);
            const float nb = nval(sq, r, p);
            const float2 er = csub(D, Xv);
            x2 += __fdividef(er.x * er.x + er.y * er.y, nb + tau);
            z[small_lay(e)] = filt(Xv, D, nb);
          }
        } else {
          for (int e = threadIdx.x; e < nu * M2; e += kSmallThreads) {
            const int lu = dm2.div(e), p = e - lu * M2, u = u0 + lu;
            const bool self = u == 0 || 2 * u == M1;
            const int sA = 2 * lu, sB = self ? sA : sA + 1, rB = self ? u : M1 - u;
            const int qi = u == 0 ? (p == 0 ? 0 : M2 - p) : M2 - 1 - p;
            if (self && p > qi) continue;
            const int ek = small_lay(sA * M2 + p), ep = small_lay(sB * M2 + qi);
            const float2 Zk = z[ek], Zp = z[ep];
            const float2 Dk = dval(sA, u, p);
            const float nk = nval(sA, u, p);
            if (u == 0 && p == 0) {   // k = 0 and k = M, both real
              const float X0 = Zk.x + Zk.y, XM = Zk.x - Zk.y, nM = __ldg(q.nyq + st.g.c);
              const float e0 = Dk.x - X0, eM = Dk.y - XM;
              x2 += __fdividef(e0 * e0, nk + tau) + __fdividef(eM * eM, nM + tau);
              const float Y0 = filt(make_float2(X0, 0.f), make_float2(Dk.x, 0.f), nk).x;
              const float YM = filt(make_float2(XM, 0.f), make_float2(Dk.y, 0.f), nM).x;
              z[ek] = make_float2(Y0 + YM, Y0 - YM);
              continue;
            }
            const float2 Dp = dval(sB, rB, qi);
            const float np = nval(sB, rB, qi);
            const float2 w = cmul(small_ld<kCache>(t_pa + u), small_ld<kCache>(t_pb + p));   // w_{2M}^k
            const float2 E = cscale(cadd(Zk, cconj(Zp)), 0.5f);
            const float2 O = cscale(mul_i<-1>(csub(Zk, cconj(Zp))), 0.5f);
            const float2 wO = cmul(w, O);
            const float2 Xk = cadd(E, wO), Xp = cconj(csub(E, wO));
            const bool same = self && qi == p;
            const float2 e1 = csub(Dk, Xk), e2 = csub(Dp, Xp);
            float t = __fdividef(e1.x * e1.x + e1.y * e1.y, nk + tau);
            if (!same) t += __fdividef(e2.x * e2.x + e2.y * e2.y, np + tau);
            x2 += 2.f * t;
            const float2 Yk = filt(Xk, Dk, nk), Yp = filt(Xp, Dp, np);
            const float2 Sm = cadd(Yk, cconj(Yp)), Tw = mul_i<+1>(cmulc(csub(Yk, cconj(Yp)), w));
            z[ek] = cadd(Sm, Tw);
            if (!same) z[ep] = cconj(csub(Sm, Tw));
          }
        }
        if (q.chi2) {   // FP32 within a warp, FP64 across warps and CTAs
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) x2 += __shfl_down_sync(0xffffffffu, x2, o);
          if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x2;
        }
        __syncthreads();
        // the peers' columns arrive in B, which no CTA touches between the two exchanges
        const float2* r = small_dft<+1, true, kCache>(z, z == A ? X : A, M2, st.g.nr2, st.g.rad2, t_row, 2 * nu);
        for (int e = threadIdx.x; e < 2 * nu * M2; e += kSmallThreads) {
          const int sq = dm2.div(e), j2 = e - sq * M2, u = u0 + (sq >> 1);
          if ((sq & 1) && (u == 0 || 2 * u == M1)) continue;
          const int k1 = row_of(sq);
          const float2 v = cmulc(r[small_lay(e)], big(k1 * j2));
          const int own = dcwf.div(j2), c = j2 - own * cw;
          const int ow = min(cw, M2 - own * cw);            // the owner's tile stride
          *cl.map_shared_rank(B + k1 * ow + c, own) = v;
        }
      }
      cl.sync();
      // the last warp adds the CTA's chi^2 while the others are in the column DFTs
      if (q.chi2 && nu > 0 && threadIdx.x >= kSmallThreads - 32) {
        const int lane = threadIdx.x & 31;
        double s = lane < kSmallThreads / 32 ? f32_to_f64(red[lane]) : 0.0;
#pragma unroll
        for (int o = kSmallThreads / 64; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) atomicAdd(q.chi2 + it, s * st.inv_nd);
      }
      // ---- inverse column DFTs, P^T T^-1 t
      if (width > 0) {
        const float2* t = small_dft<+1, false, kCache>(B, A, M1, st.g.nr1, st.g.rad1, t_col, width);
        const uint64_t pol = l2_policy_evict_last();
        const int64_t stride = acc_stride_of(q.n_pix, NC);
        const int ne = M1 * width;
        for (int e0 = threadIdx.x & ~31; e0 < ne; e0 += kSmallThreads) {   // warp-uniform
          const int e = e0 + (threadIdx.x & 31);
          int px[2] = {-1, -1};
          float a[2][3] = {};
          if (e < ne) {
            int64_t s = 0;
            if constexpr (!kCache) {
              const int j1 = dcw.div(e), c = e - j1 * width;
              s = off + ((int64_t)j1 * M2 + j0 + c) * nh;
            }
            const float2 v = t[e];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              if (h >= nh) continue;
              a[h][0] = h ? v.y : v.x;
              if constexpr (kCache) {
                px[h] = c_pix[2 * e + h];
                if constexpr (NC == 3) {
                  a[h][1] = a[h][0] * c_cos[2 * e + h];
                  a[h][2] = a[h][0] * c_sin[2 * e + h];
                }
              } else {
                px[h] = __ldg(q.pix + s + h);
                if constexpr (NC == 3) {
                  a[h][1] = a[h][0] * weight(q.cosw, s + h);
                  a[h][2] = a[h][0] * weight(q.sinw, s + h);
                }
              }
            }
          }
          // equal pixels of an element's two samples, then of two neighbouring elements, add
          // up before the reduction
          bool one = nh == 1;
          if (nh == 2 && px[0] == px[1]) {
#pragma unroll
            for (int k = 0; k < NC; ++k) a[0][k] += a[1][k];
            px[1] = -1;
            one = true;
          }
          const int key = one ? px[0] : -2 - e;   // never equal to another lane's unless one pixel
          const int other = __shfl_xor_sync(0xffffffffu, key, 1);
          const bool pair = one && other == key;
#pragma unroll
          for (int k = 0; k < NC; ++k) {
            const float o = __shfl_down_sync(0xffffffffu, a[0][k], 1);
            if (pair) a[0][k] += o;
          }
          if (pair && (threadIdx.x & 1)) px[0] = -1;
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (px[h] >= 0) {
#pragma unroll
              for (int k = 0; k < NC; ++k) red_add_f64(q.acc + k * stride + px[h], f32_to_f64(a[h][k]), pol);
            }
        }
      }
      // the next chunk's (or iteration's) gather and first exchange write A and X only; B is
      // free again after its own columns are binned
      __syncthreads();
    }
    sync_all();
    // ---- map step: groups of 32 pixels over all warps of the grid, CTA by CTA first (FP64
    // arithmetic is slow, and few pixels on one SM would queue for it)
    {
      const int64_t stride = acc_stride_of(q.n_pix, NC);
      double* out = it == q.n_iter - 1 ? q.map_out : nullptr;
      for (int64_t p = 32 * ((int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) + (threadIdx.x & 31); p < q.n_pix;
           p += (int64_t)gridDim.x * kSmallThreads) {
        double a[NC], m[NC], w[NC == 3 ? 6 : 1];
#pragma unroll
        for (int k = 0; k < NC; ++k) a[k] = __ldcg(q.acc + k * stride + p);
#pragma unroll
        for (int k = 0; k < (NC == 3 ? 6 : 1); ++k) w[k] = __ldg(q.W + (NC == 3 ? 6 : 1) * p + k);
        // every load before the first store
#pragma unroll
        for (int k = 0; k < NC; ++k) q.acc[k * stride + p] = 0.0;
        if constexpr (NC == 1) {
          m[0] = w[0] * a[0];
          reinterpret_cast<float*>(q.map4)[p] = (float)m[0];
        } else {
          m[0] = w[0] * a[0] + w[1] * a[1] + w[2] * a[2];
          m[1] = w[1] * a[0] + w[3] * a[1] + w[4] * a[2];
          m[2] = w[2] * a[0] + w[4] * a[1] + w[5] * a[2];
          reinterpret_cast<float4*>(q.map4)[p] = make_float4((float)m[0], (float)m[1], (float)m[2], 0.f);
        }
        if (out)
#pragma unroll
          for (int k = 0; k < NC; ++k) out[NC * p + k] = m[k];
      }
    }
    if (it + 1 < q.n_iter) sync_all();
  }
  cl.sync();   // no CTA leaves while a peer may still write into its shared memory
}

// ------------------------------------------------------------------------ host side
// Words of one work buffer for a chunk of M1 x M2 over S CTAs.
static int small_tile_words(const ChunkDesc& d, int S) {
  const int cw = (d.M2 + S - 1) / S, upc = (d.M1 / 2 + 1 + S - 1) / S;
  const int col = d.M1 * cw, row = 2 * upc * d.M2 + ((2 * upc * d.M2) >> 4) + 1;
  return ((col > row ? col : row) + 3) & ~3;
}

static int small_table_words(const ChunkDesc& d, int log_lo) {
  return (3 * (d.M1 + d.M2) + (1 << log_lo) + (d.M >> log_lo) + 1 + 3) & ~3;
}

static size_t small_smem(int tile, int tables, int ncomp, bool cache) {
  size_t w = 3 * sizeof(float2) * (size_t)tile;
  if (cache) w += (size_t)tile * (8 + 4 + 2 * 4 * (ncomp == 3 ? 3 : 1)) + sizeof(float2) * (size_t)tables;
  return w;
}

static void small_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, int S, int grid, size_t smem,
                         cudaStream_t st) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(grid);
  cfg->blockDim = dim3(kSmallThreads);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = S;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeCooperative;
  at[1].val.cooperative = 1;
  cfg->attrs = at;
  cfg->numAttrs = 2;
}

// Clusters of S CTAs of kernel k that fit the device at once (0 when the buffers don't fit);
// cached, because the query takes tens of microseconds.
template <typename K>
static cudaError_t small_clusters(K k, int S, size_t smem, int* n) {
  static std::mutex mu;
  static std::map<std::tuple<const void*, int, int, size_t>, int> known;
  *n = 0;
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const auto key = std::make_tuple(reinterpret_cast<const void*>(k), dev, S, smem);
  {
    std::lock_guard<std::mutex> g(mu);
    auto it = known.find(key);
    if (it != known.end()) { *n = it->second; return cudaSuccess; }
    if (known.size() >= 4096) known.clear();
  }
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa;
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
  if (e != cudaSuccess) return e;
  const int most = optin - (int)fa.sharedSizeBytes;
  if (smem > (size_t)most) return cudaSuccess;
  if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess) return e;
  if (S > 8 && (e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
    return e;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[2];
  small_config(&cfg, at, S, S, smem, nullptr);
  if ((e = cudaOccupancyMaxActiveClusters(n, k, &cfg)) != cudaSuccess) return e;
  std::lock_guard<std::mutex> g(mu);
  known[key] = *n;
  return cudaSuccess;
}

// Words of a work buffer times a cluster's turns up to which a plan takes this path.  Measured
// per iteration against the three-kernel path (chunks x samples): power-of-two lengths, T-only,
// 4 x 2^15 (2450 words) 16.3 against 24.4 us, 8 x 2^16 (4900) 23.2 / 28.1, 4 x 2^17 (9700)
// 44.7 / 28.5; IQU 18.7 / 28.3, 32.0 / 32.2, 52.2 / 34.6 (clusters of 8).  Clusters of 16, where
// they fit (about four at once): IQU 4 x 2^15 16.3, 4 x 2^16 18.9 us, T-only 4 x 2^17 22.9.  General
// lengths, whose three kernels are slower, IQU: 12 chunks of 1500 to 12000 samples 15.8 / 40.9, 4 of 20000 to 90000 (5600
// words) 46.3 / 53.1, with clusters of 16 25.6.
static int small_limit(bool general, int ncomp) {
  return general ? 6144 : ncomp == 1 ? 5120 : 4096;
}

// Pixels up to which a plan takes this path: its map step runs on its own CTAs, at about 3.2 ns a
// pixel and CTA (IQU; T-only 0.55), against the whole GPU in a launch of its own; and beyond the
// second limits the sums, weights and map no longer stay in L2.  Per iteration against the
// three-kernel path, IQU, 2^12 samples (8 CTAs): 2^15 pixels 21.9 / 23.0 us, 2^16 35.1 / 24.0, 2^20
// 437 / 51.7; 2^15 samples (16 CTAs): 2^16 pixels 26.1 / 28.5, 2^17 39.4 / 31.2; 4 x 2^15 samples (64 CTAs):
// 2^18 pixels 28.0 / 35.0, 2^19 41.5 / 40.3, 2^20 148 / 57.2; 12 ragged chunks: 2^19 pixels 31.0 / 49.7,
// 2^20 99.5 / 71.1.  T-only: 2^12 samples: 2^17 pixels 17.4 / 23.0, 2^18 26.4 / 23.0; 4 x 2^15 samples: 2^20
// pixels 23.4 / 32.7, 2^21 32.5 / 35.5, 2^22 186 / 48.3; 40 x 2^13: 2^21 pixels 30.8 / 39.6, 2^22 100 / 51.1.
static int64_t small_pixels(int ctas, int ncomp) {
  const int64_t per_cta = (int64_t)ctas * (ncomp == 1 ? 20480 : 4096), l2 = ncomp == 1 ? 1 << 21 : 1 << 19;
  return per_cta < l2 ? per_cta : l2;
}

template <int NC>
static cudaError_t small_plan_nc(const mm_plan_s* p, SmallShape* out) {
  *out = SmallShape{};
  const int limit = small_limit(p->n_gen > 0, NC);
  int tables = 0;
  for (int c = 0; c < p->n_chunks; ++c) {
    const ChunkDesc& d = p->h_desc[c];
    if (d.M > 16 * limit) return cudaSuccess;
    tables = std::max(tables, small_table_words(d, p->groups[d.grp].log_lo));
  }
  auto largest = [&](int S) {
    int tile = 0;
    for (int c = 0; c < p->n_chunks; ++c) tile = std::max(tile, small_tile_words(p->h_desc[c], S));
    return tile;
  };
  SmallShape best;
  // clusters of 16 for chunks whose share of 8 CTAs is not tiny (below, the larger cluster's
  // barriers cost more than the halved tiles save: 4 x 2^12 10.4 us against 11.4)
  for (int S = largest(8) >= 512 ? 16 : 8; S >= 1; S /= 2) {
    const int tile = largest(S);
    int n = 0;
    if (tile > limit) break;   // smaller clusters hold larger tiles
    // the largest cluster size whose clusters keep a chunk each; else the one with the most clusters
    cudaError_t e = small_clusters(k_small<NC, true>, S, small_smem(tile, tables, NC, true), &n);
    if (e != cudaSuccess) return e;
    if (n >= p->n_chunks) {
      best = SmallShape{S, p->n_chunks, tile, tables, 1};
      break;
    }
    if ((e = small_clusters(k_small<NC, false>, S, small_smem(tile, tables, NC, false), &n)) != cudaSuccess) return e;
    const int cl = std::min(n, p->n_chunks);
    if (cl > best.clusters) best = SmallShape{S, cl, tile, tables, 0};
  }
  if (best.clusters > 0 &&
      (int64_t)best.tile * ((p->n_chunks + best.clusters - 1) / best.clusters) <= limit &&
      p->n_pix <= small_pixels(best.S * best.clusters, NC))
    *out = best;
  return cudaSuccess;
}

cudaError_t small_shape(const mm_plan_s* p, SmallShape* out) {
  return p->ncomp == 3 ? small_plan_nc<3>(p, out) : small_plan_nc<1>(p, out);
}

template <int NC>
static cudaError_t launch_small_nc(const mm_plan_s* p, const double* lambdas, int n_iter, double* map_out,
                                   double* chi2, cudaStream_t st) {
  const SmallShape& s = p->small;
  SmallParams q;
  q.rec = p->small_rec;
  q.desc = p->d_desc;
  q.n_chunks = p->n_chunks;
  q.tile = s.tile;
  q.tables = s.tables;
  q.pix = p->pix;
  q.cosw = p->cosw;
  q.sinw = p->sinw;
  q.half_w = p->wdtype == MM_W_F16;
  q.dtab = p->dtab;
  q.nbar = p->nbar;
  q.nyq = p->nyq;
  q.W = p->W;
  q.acc = p->acc;
  q.map4 = p->map4;
  q.n_pix = p->n_pix;
  q.bar = p->small_bar;
  q.fault = p->fault;
  q.n_polls = p->wait_polls;
  for (int i0 = 0; i0 < n_iter; i0 += kSmallLambdas) {
    q.n_iter = n_iter - i0 < kSmallLambdas ? n_iter - i0 : kSmallLambdas;
    for (int i = 0; i < q.n_iter; ++i) q.lambda[i] = lambdas[i0 + i];
    q.map_out = i0 + q.n_iter == n_iter ? map_out : nullptr;
    q.chi2 = chi2 ? chi2 + i0 : nullptr;
    cudaError_t e;
    if (s.clusters > 1 && (e = cudaMemsetAsync(p->small_bar, 0, sizeof(unsigned), st)) != cudaSuccess) return e;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[2];
    small_config(&cfg, at, s.S, s.S * s.clusters, small_smem(s.tile, s.tables, NC, s.cache != 0), st);
    e = s.cache ? cudaLaunchKernelEx(&cfg, k_small<NC, true>, q) : cudaLaunchKernelEx(&cfg, k_small<NC, false>, q);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

cudaError_t launch_small(const mm_plan_s* p, const double* lambdas, int n_iter, double* map_out, double* chi2,
                         cudaStream_t st) {
  return p->ncomp == 3 ? launch_small_nc<3>(p, lambdas, n_iter, map_out, chi2, st)
                       : launch_small_nc<1>(p, lambdas, n_iter, map_out, chi2, st);
}

}  // namespace mm
