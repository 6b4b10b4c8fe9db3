// Attention over the stored reconstruction R_phi(K, V) (Sections 3.2-3.3).
// Prefill: causal attention of the newest L queries over all T tokens.
// Decode: L = 1, split over the tokens, partials merged by log-sum-exp.
#include <math.h>

#include "kvq_internal.cuh"
#include "reconstruct.cuh"

namespace kvq {
namespace {

constexpr int kTile = 64;       // tokens per shared-memory tile
constexpr int kThreads = 256;

// Split-K partials of (b, q head): kMaxSplits rows of (m, l, o[D]).
__device__ __forceinline__ float* ws_row(const Geom& g, int b, int hq) {
  return reinterpret_cast<float*>(g.pl[KVQ_PLANE_WORKSPACE].p) +
         ((int64_t)b * g.Hq + hq) * kMaxSplits * (g.D + kWsStride);
}

__device__ __forceinline__ unsigned code_at(const uint8_t* row, int d, int bits) {
  const int bit = d * bits;
  return (row[bit >> 3] >> (bit & 7)) & ((1u << bits) - 1);
}

// KVarN: tokens [t0, t0 + n) of one (b, h) in the rotated basis into dst
// [n][ld] (fp32): the coded rows are stored rotated, the full-precision rows
// (sinks, staged) are rotated forward.  which = 0 keys, 1 values; T = tokens
// stored; tokens from `end` on are zero.
__device__ void kvarn_rows(const Geom& g, int which, int b, int h, int t0, int n, int end, int T,
                           float* dst, int ld, float inv_sqrt_d) {
  const int D = g.D, G = g.G;
  const int bits = which ? g.vb : g.kb;
  const int P_CODES = which ? KVQ_PLANE_V_CODES : KVQ_PLANE_K_CODES;
  const int P_SCALE = which ? KVQ_PLANE_V_SCALE : KVQ_PLANE_K_SCALE;
  const int P_ZERO = which ? KVQ_PLANE_V_ZERO : KVQ_PLANE_K_ZERO;
  const int P_FULL = which ? KVQ_PLANE_V_FULL : KVQ_PLANE_K_FULL;
  const int P_PEND = which ? KVQ_PLANE_V_PEND : KVQ_PLANE_K_PEND;
  const int P_ROW = which ? KVQ_PLANE_V_ROW : KVQ_PLANE_K_ROW;
  const int P_COL = which ? KVQ_PLANE_V_COL : KVQ_PLANE_K_COL;
  const int nbq = kvarn_nblocks(T, g.S, G) * G;
  for (int i = threadIdx.x; i < n * D; i += blockDim.x) {
    const int r = i / D, d = i % D, t = t0 + r;
    float val = 0.f;
    if (t < end) {
      if (t < g.S) {
        val = ld_act(g.pl[P_FULL].p, plane_index(g.pl[P_FULL], b, h, g.H, t, d), g.act);
      } else if (t - g.S < nbq) {
        const int q = t - g.S;
        unsigned c = code_at(plane_ptr<uint8_t>(g, P_CODES, b, h, q), d, bits);
        float s = __half2float(*plane_ptr<__half>(g, P_SCALE, b, h, q, d / G));
        float m = __half2float(*plane_ptr<__half>(g, P_ZERO, b, h, q, d / G));
        float rr = __half2float(*plane_ptr<__half>(g, P_ROW, b, h, 0, q));
        float cc = __half2float(*plane_ptr<__half>(g, P_COL, b, h, q / G, d));
        val = rr * cc * ((float)c * s + m);
      } else {
        val = ld_act(g.pl[P_PEND].p, plane_index(g.pl[P_PEND], b, h, g.H, (t - g.S) % G, d), g.act);
      }
    }
    dst[r * ld + d] = val;
  }
  if (!(t0 >= g.S && t0 + n <= g.S + nbq)) {
    __syncthreads();
    for (int hs = 1; hs < D; hs <<= 1) {
      for (int p = threadIdx.x; p < n * D / 2; p += blockDim.x) {
        const int r = p / (D / 2), k = p % (D / 2), t = t0 + r;
        if (t >= T || (t >= g.S && t - g.S < nbq)) continue;
        const int j = (k / hs) * 2 * hs + (k % hs);
        float a = dst[r * ld + j], c = dst[r * ld + j + hs];
        dst[r * ld + j] = a + c;
        dst[r * ld + j + hs] = a - c;
      }
      __syncthreads();
    }
    for (int i = threadIdx.x; i < n * D; i += blockDim.x) {
      const int r = i / D, t = t0 + r;
      if (t < T && !(t >= g.S && t - g.S < nbq)) dst[r * ld + i % D] *= inv_sqrt_d;
    }
  }
}

// The other formats: 8 channels of a token per thread and step; tokens from `end` on
// are zero.
template <int D>
__device__ __forceinline__ void dequant_rows(const Geom& g, int which, int b, int h, int t0, int n,
                                             int end, int tq, float* dst, int ld) {
  const bool f32 = g.act == KVQ_F32;
  const int P_FULL = which ? KVQ_PLANE_V_FULL : KVQ_PLANE_K_FULL;
  for (int i = threadIdx.x; i < n * (D / 8); i += kThreads) {
    const int r = i / (D / 8), c = i % (D / 8), t = t0 + r;
    float4* d4 = reinterpret_cast<float4*>(dst + r * ld + 8 * c);
    if (f32 && t < end && (g.fmt == KVQ_FMT_FLOAT || (g.fmt == KVQ_FMT_KIVI && t >= tq))) {
      const float4* src = reinterpret_cast<const float4*>(
          plane_ptr<float>(g, P_FULL, b, h, g.fmt == KVQ_FMT_KIVI ? t % g.ring : t, 8 * c));
      d4[0] = src[0];
      d4[1] = src[1];
    } else {
      float v[8];
      deq8(g, which, b, h, t, c, end, tq, v);
      d4[0] = make_float4(v[0], v[1], v[2], v[3]);
      d4[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
  }
}

// Affine and symmetric caches: this thread's part of a tile as stored, NI = D / 32
// chunks of 8 channels (chunk threadIdx.x + 256 i, rows of D / 8 chunks), so that the
// next tile's loads are in flight while a tile is multiplied.
template <int D>
struct PackedChunks {
  static constexpr int NI = kTile * (D / 8) / kThreads;
  uint64_t w[NI];
  __half s[NI], z[NI];
  __device__ __forceinline__ void load(const Geom& g, int which, int b, int h, int t0, int n, int T,
                                       int lg) {
    const int bits = which ? g.vb : g.kb;
    const uint8_t* codes = plane_ptr<uint8_t>(g, which ? KVQ_PLANE_V_CODES : KVQ_PLANE_K_CODES, b, h, 0);
    const __half* sp = plane_ptr<__half>(g, which ? KVQ_PLANE_V_SCALE : KVQ_PLANE_K_SCALE, b, h, 0);
    const __half* zp = g.fmt == KVQ_FMT_SYMMETRIC
                           ? nullptr : plane_ptr<__half>(g, which ? KVQ_PLANE_V_ZERO : KVQ_PLANE_K_ZERO, b, h, 0);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int idx = threadIdx.x + kThreads * i, c = idx % (D / 8), t = t0 + idx / (D / 8);
      w[i] = 0;
      s[i] = z[i] = __half(0.f);
      if (idx / (D / 8) >= n || t >= T) continue;
      const uint8_t* p = codes + (int64_t)t * (D * bits / 8) + c * bits;
      w[i] = bits == 4 ? *reinterpret_cast<const uint32_t*>(p)
           : bits == 2 ? *reinterpret_cast<const uint16_t*>(p) : *reinterpret_cast<const uint64_t*>(p);
      const int64_t m = (int64_t)t * (D >> lg) + ((8 * c) >> lg);
      s[i] = sp[m];
      if (zp) z[i] = zp[m];
    }
  }
  __device__ __forceinline__ void expand(const Geom& g, int which, int n, float* dst, int ld) const {
    const int bits = which ? g.vb : g.kb;
    const unsigned mask = (1u << bits) - 1;
    // symmetric: (code - zero) x scale, which is infinite, not NaN, where the scale is
    const int zero = g.fmt == KVQ_FMT_SYMMETRIC ? 1 << (bits - 1) : 0;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int idx = threadIdx.x + kThreads * i, c = idx % (D / 8), r = idx / (D / 8);
      if (r >= n) continue;
      const float sc = __half2float(s[i]), m = __half2float(z[i]);
      float v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e)
        v[e] = (float)((int)((unsigned)(w[i] >> (e * bits)) & mask) - zero) * sc + m;
      float4* d = reinterpret_cast<float4*>(dst + r * ld + 8 * c);
      d[0] = make_float4(v[0], v[1], v[2], v[3]);
      d[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
  }
};

// Normalised Hadamard transform of `rows` rows of D values at x [rows][ld]
// (the whole CTA; H / sqrt(D) is its own inverse).
__device__ void rotate_rows(float* x, int rows, int D, int ld, float inv_sqrt_d) {
  __syncthreads();
  for (int hs = 1; hs < D; hs <<= 1) {
    for (int p = threadIdx.x; p < rows * D / 2; p += blockDim.x) {
      const int r = p / (D / 2), k = p % (D / 2);
      const int j = (k / hs) * 2 * hs + (k % hs);
      const float a = x[r * ld + j], c = x[r * ld + j + hs];
      x[r * ld + j] = a + c;
      x[r * ld + j + hs] = a - c;
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < rows * D; i += blockDim.x) x[(i / D) * ld + i % D] *= inv_sqrt_d;
  __syncthreads();
}

// Attention in fp32 for every format, fp32 activations (prefill and decode) and
// the bf16 caches that no tensor-core decode covers.  One CTA = ROWS rows (the g
// query heads x nq queries of one (b, kv head)) over the tokens [ts, te), 64
// at a time; shared memory holds the K and V tiles, q and the scores, the
// output accumulates in registers.
//   scores: warp w has row group w % 4 and 32 of the tile's tokens, a lane one
//     token for all rows of the group (its K row read once, q broadcast);
//   softmax: 256 / ROWS threads per row;
//   P V: a thread has 4 channels of ROWS D / 1024 rows.
// These sizes are far from filling the GPU (a 512-token prompt of 4 heads is
// 0.07 GFLOP a head), so the latency of one CTA's chain of tiles bounds it: 16
// rows a CTA give 8 times the CTAs of 128 rows, and 64 rows serve where 16 are
// not needed to cover the SMs twice.  512 tokens, 4 heads of 64, fp32, affine
// 4-bit: 1142 -> 34 us, a decode step after them 24 + 10 -> 14 us.
// decode: writes (m, l, o) partials to the workspace; the last split CTA of a
// (sequence, kv head) merges them (one launch instead of two).
template <int D, int ROWS>
struct GenSmem {
  static constexpr int LDK = D + 4;                // 16-byte rows in distinct banks
  static constexpr int LDS = kTile + 4;
  float k[kTile * LDK];                            // then the output rows [ROWS][D]
  float v[kTile * D];
  float q[ROWS * D];
  float s[ROWS * LDS];
  float alpha[ROWS], m[ROWS], l[ROWS];
};

template <int D, int ROWS>
__global__ void __launch_bounds__(kThreads)
attend_generic_kernel(Geom g, const void* q, int L, float scale, void* out,
                      int nq, int splits, int decode, float inv_sqrt_d) {
  pdl_wait();
  pdl_trigger();
  using S = GenSmem<D, ROWS>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  S& sm = *reinterpret_cast<S*>(smem_raw);
  const int T = cache_tokens(g);
  const int tq = g.fmt == KVQ_FMT_KIVI ? kivi_tq(T, g.R, g.G) : T;
  const int grp = g.Hq / g.H;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // longest first (causal work grows with the position)
  const int qtile = gridDim.x / splits - 1 - blockIdx.x / splits, split = blockIdx.x % splits;
  const int hkv = blockIdx.y, b = blockIdx.z;
  const int q0 = qtile * nq;            // first query of this CTA
  const int nql = min(nq, L - q0);
  const int pos_first = T - L + q0;     // absolute position of query q0
  // tokens of this split
  int ts = 0, te = pos_first + nql;
  if (decode) split_range(T, splits, split, 32, &ts, &te);
  auto row_pos = [&](int r) {           // last token that row r sees, -1 for padding rows
    const int hl = r / nq, qi = r % nq;
    return hl < grp && qi < nql ? pos_first + qi : -1;
  };
  const bool kvarn = g.fmt == KVQ_FMT_KVARN;
  const bool packed = g.fmt == KVQ_FMT_AFFINE || g.fmt == KVQ_FMT_SYMMETRIC;
  const int lg = __ffs(g.G) - 1;                  // G is a power of two
  PackedChunks<D> pk, pv;
  if (packed && ts < te) {
    pk.load(g, 0, b, hkv, ts, te - ts, T, lg);
    pv.load(g, 1, b, hkv, ts, te - ts, T, lg);
  }
  for (int i = threadIdx.x; i < ROWS * D; i += kThreads) {
    const int r = i / D, d = i % D;
    const int hl = r / nq, qi = r % nq;
    float v = 0.f;
    if (hl < grp && qi < nql)
      v = ld_act(q, (((int64_t)b * g.Hq + hkv * grp + hl) * L + q0 + qi) * D + d, g.act);
    sm.q[i] = v;
  }
  if (kvarn) rotate_rows(sm.q, ROWS, D, D, inv_sqrt_d);     // queries into the rotated basis

  constexpr int RS = ROWS / 4;                    // score rows of a thread
  constexpr int TPR = kThreads / ROWS;            // softmax threads per row
  constexpr int NRG = 4 * kThreads / D;           // P V row groups
  constexpr int RO = ROWS / NRG;                  // P V rows of a thread
  static_assert(RO >= 1, "every P V thread has a row");
  const int srow = (warp & 3) * RS, stok = (warp >> 2) * 32 + lane;
  int spos[RS];
#pragma unroll
  for (int k = 0; k < RS; ++k) spos[k] = row_pos(srow + k);
  const int xrow = threadIdx.x / TPR, xsub = threadIdx.x % TPR;
  float m_run = -INFINITY, l_run = 0.f;           // l_run: this thread's share
  const int od = threadIdx.x % (D / 4), orow = threadIdx.x / (D / 4);
  float4 acc[RO];
#pragma unroll
  for (int k = 0; k < RO; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);

  for (int t0 = ts; t0 < te; t0 += kTile) {
    const int n = min(kTile, te - t0);
    // rows read below: those past the last token are zero, not the next tokens
    // (weight 0 times an infinite value is NaN)
    const int n4 = (n + 3) & ~3;
    __syncthreads();                              // previous tile consumed (and q stored)
    if (packed) {
      pk.expand(g, 0, n4, sm.k, S::LDK);
      pv.expand(g, 1, n4, sm.v, D);
      if (t0 + kTile < te) {
        pk.load(g, 0, b, hkv, t0 + kTile, te - t0 - kTile, T, lg);
        pv.load(g, 1, b, hkv, t0 + kTile, te - t0 - kTile, T, lg);
      }
    } else if (kvarn) {
      kvarn_rows(g, 0, b, hkv, t0, n4, te, T, sm.k, S::LDK, inv_sqrt_d);
      kvarn_rows(g, 1, b, hkv, t0, n4, te, T, sm.v, D, inv_sqrt_d);
    } else {
      dequant_rows<D>(g, 0, b, hkv, t0, n4, te, tq, sm.k, S::LDK);
      dequant_rows<D>(g, 1, b, hkv, t0, n4, te, tq, sm.v, D);
    }
    __syncthreads();
    if ((warp >> 2) * 32 < n4) {
      float sc[RS];
#pragma unroll
      for (int k = 0; k < RS; ++k) sc[k] = 0.f;
      const float4* kr = reinterpret_cast<const float4*>(sm.k + stok * S::LDK);
#pragma unroll 4
      for (int d = 0; d < D / 4; ++d) {
        const float4 kv = kr[d];
#pragma unroll
        for (int k = 0; k < RS; ++k) {
          const float4 qv = reinterpret_cast<const float4*>(sm.q + (srow + k) * D)[d];
          sc[k] = fmaf(qv.x, kv.x, sc[k]);
          sc[k] = fmaf(qv.y, kv.y, sc[k]);
          sc[k] = fmaf(qv.z, kv.z, sc[k]);
          sc[k] = fmaf(qv.w, kv.w, sc[k]);
        }
      }
#pragma unroll
      for (int k = 0; k < RS; ++k)
        sm.s[(srow + k) * S::LDS + stok] =
            stok < n && t0 + stok <= spos[k] ? sc[k] * scale : -INFINITY;
    }
    __syncthreads();
    {
      float mx = -INFINITY;
      float* srw = sm.s + xrow * S::LDS;
      for (int j = xsub; j < n; j += TPR) mx = fmaxf(mx, srw[j]);
#pragma unroll
      for (int o = TPR / 2; o >= 1; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float mn = fmaxf(m_run, mx);
      const float alpha = mn == -INFINITY ? 1.f : expf(m_run - mn);
      float sum = 0.f;
      for (int j = xsub; j < n4; j += TPR) {
        const float sv = srw[j];
        const float p = sv == -INFINITY ? 0.f : expf(sv - mn);
        srw[j] = p;
        sum += p;
      }
      l_run = l_run * alpha + sum;
      m_run = mn;
      if (xsub == 0) sm.alpha[xrow] = alpha;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < RO; ++k) {
      const float f = sm.alpha[orow + NRG * k];
      acc[k].x *= f; acc[k].y *= f; acc[k].z *= f; acc[k].w *= f;
    }
#pragma unroll 2
    for (int j = 0; j < n4; j += 4) {
      float4 vv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) vv[u] = reinterpret_cast<const float4*>(sm.v + (j + u) * D)[od];
#pragma unroll
      for (int k = 0; k < RO; ++k) {
        const float4 p = *reinterpret_cast<const float4*>(sm.s + (orow + NRG * k) * S::LDS + j);
        const float pu[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          acc[k].x = fmaf(pu[u], vv[u].x, acc[k].x);
          acc[k].y = fmaf(pu[u], vv[u].y, acc[k].y);
          acc[k].z = fmaf(pu[u], vv[u].z, acc[k].z);
          acc[k].w = fmaf(pu[u], vv[u].w, acc[k].w);
        }
      }
    }
  }
#pragma unroll
  for (int o = TPR / 2; o >= 1; o >>= 1) l_run += __shfl_xor_sync(0xffffffffu, l_run, o);
  if (xsub == 0) {
    sm.m[xrow] = m_run;
    sm.l[xrow] = l_run;
  }
  __syncthreads();                                // K tile consumed: output rows over it
  float* os = sm.k;
#pragma unroll
  for (int k = 0; k < RO; ++k)
    reinterpret_cast<float4*>(os + (orow + NRG * k) * D)[od] = acc[k];
  __syncthreads();
  if (kvarn) rotate_rows(os, ROWS, D, D, inv_sqrt_d);       // back to the original basis
  if (!decode) {
    for (int i = threadIdx.x; i < ROWS * D; i += kThreads) {
      const int r = i / D, d = i % D;
      const int hl = r / nq, qi = r % nq;
      if (hl >= grp || qi >= nql) continue;
      st_act(out, (((int64_t)b * g.Hq + hkv * grp + hl) * L + q0 + qi) * D + d, os[i] / sm.l[r],
             g.act);
    }
    return;
  }
  for (int i = threadIdx.x; i < grp * (D + kWsStride); i += kThreads) {
    const int r = i / (D + kWsStride), c = i % (D + kWsStride);   // nq == 1 in decode
    ws_row(g, b, hkv * grp + r)[(int64_t)split * (D + kWsStride) + c] =
        c == 0 ? sm.m[r] : c == 1 ? sm.l[r] : os[r * D + c - 2];
  }
  // the last split CTA of this (sequence, kv head) merges:
  // o = sum_s e^(m_s - M) o_s / sum_s e^(m_s - M) l_s
  __shared__ int last_cta;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last_cta = atomicAdd(&g.counters[b * g.H + hkv], 1u) == (unsigned)splits - 1;
  }
  __syncthreads();
  if (!last_cta) return;
  __threadfence();
  for (int hl = warp; hl < grp; hl += kThreads / 32) {
    const float* w = ws_row(g, b, hkv * grp + hl);
    const float ms = lane < splits ? __ldcg(w + (int64_t)lane * (D + kWsStride)) : -INFINITY;
    const float ls = lane < splits ? __ldcg(w + (int64_t)lane * (D + kWsStride) + 1) : 0.f;
    float M = ms;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    const float f = ms == -INFINITY ? 0.f : expf(ms - M);
    float Ls = f * ls;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) Ls += __shfl_xor_sync(0xffffffffu, Ls, o);
    float o[D / 32];
#pragma unroll
    for (int k = 0; k < D / 32; ++k) o[k] = 0.f;
#pragma unroll 4
    for (int i = 0; i < splits; ++i) {
      const float fi = __shfl_sync(0xffffffffu, f, i);
      const float* wi = w + (int64_t)i * (D + kWsStride) + 2 + lane;
#pragma unroll
      for (int k = 0; k < D / 32; ++k) o[k] = fmaf(fi, __ldcg(wi + 32 * k), o[k]);
    }
#pragma unroll
    for (int k = 0; k < D / 32; ++k)
      st_act(out, ((int64_t)b * g.Hq + hkv * grp + hl) * D + lane + 32 * k, o[k] / Ls, g.act);
  }
  if (threadIdx.x == 0) g.counters[b * g.H + hkv] = 0;   // ready for the next call
}

template <int D, int ROWS>
cudaError_t launch_generic(const Geom& g, const void* q, int L, float scale, void* out,
                           bool decode, cudaStream_t s) {
  auto kern = attend_generic_kernel<D, ROWS>;
  const int sm = (int)sizeof(GenSmem<D, ROWS>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  if (e != cudaSuccess) return e;
  const int nq = decode ? 1 : ROWS / (g.Hq / g.H), splits = decode ? g.splits : 1;
  const float inv_sqrt_d = (float)(1.0 / sqrt((double)D));
  launch_pdl(kern, dim3((L + nq - 1) / nq * splits, g.H, g.B), dim3(kThreads), (size_t)sm, s, g, q,
             L, scale, out, nq, splits, decode ? 1 : 0, inv_sqrt_d);
  return cudaGetLastError();
}

template <int D>
cudaError_t launch_generic_d(const Geom& g, const void* q, int L, float scale, void* out,
                             bool decode, cudaStream_t s) {
  const int64_t ctas64 = (int64_t)((L * (g.Hq / g.H) + 63) / 64) * g.H * g.B;
  return !decode && ctas64 >= 2 * num_sms()
             ? launch_generic<D, 64>(g, q, L, scale, out, decode, s)
             : launch_generic<D, 16>(g, q, L, scale, out, decode, s);
}

// ---------------------------------------------------------------------------
// KVarN decode attention in the rotated basis (Section 3.1: coded tokens are
// stored as r_t c_j (s code + m) after the normalised Hadamard rotation).
// One CTA = (split, kv head, sequence), 8 warps, each warp a contiguous part
// of the split; lane l holds channels [NS l, NS l + NS), NS = D / 32.  The
// queries are rotated once (in registers); a coded token's score is
//   r_t (s_t sum_j q'_j code_j + m_t sum_j q'_j),  q' = q_rot c_block,
// refolded when the token block changes (a lane's channels lie in one group);
// sinks and staged tokens are rotated forward in registers.  The values
// accumulate in the rotated basis; the split's output is rotated back before
// its (m, l, o) partial goes to the workspace, and the last split CTA of a
// (sequence, kv head) to finish merges the partials into the output.
// ---------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ void fwht_contig(float (&x)[D / 32], int lane, float inv_sqrt_d) {
  constexpr int NS = D / 32;
#pragma unroll
  for (int h = 1; h < NS; h <<= 1)
#pragma unroll
    for (int i = 0; i < NS; ++i)
      if (!(i & h)) {
        const float a = x[i], c = x[i + h];
        x[i] = a + c;
        x[i + h] = a - c;
      }
#pragma unroll
  for (int lh = 1; lh < 32; lh <<= 1)
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      const float y = __shfl_xor_sync(0xffffffffu, x[i], lh);
      x[i] = (lane & lh) ? y - x[i] : x[i] + y;
    }
#pragma unroll
  for (int i = 0; i < NS; ++i) x[i] *= inv_sqrt_d;
}

// NS codes of `bits` bits of this lane's channels from a packed row
__device__ __forceinline__ uint32_t lane_codes(const uint8_t* row, int lane, int ns, int bits) {
  const int bit = ns * bits * lane;
  return __ldg(reinterpret_cast<const uint32_t*>(row) + (bit >> 5)) >> (bit & 31);
}

template <int D, int GM>
__global__ void __launch_bounds__(256)
attend_kvarn_decode_kernel(Geom g, const __nv_bfloat16* __restrict__ q, float scale,
                           float inv_sqrt_d, void* out) {
  pdl_wait();
  pdl_trigger();
  constexpr int NS = D / 32;
  extern __shared__ float ksm[];                 // [8 warps][GM][D + 2]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int split = blockIdx.x, hkv = blockIdx.y, b = blockIdx.z;
  const int grp = g.Hq / g.H, G = g.G, S = g.S;
  const int T = cache_tokens(g);
  const int nbq = kvarn_nblocks(T, S, G) * G;
  int ts, te;
  split_range(T, g.splits, split, G, &ts, &te);
  const float c2 = scale * 1.4426950408889634f;   // scores in log2 units
  // rotated queries, pre-scaled
  float qr[GM][NS];
#pragma unroll
  for (int h = 0; h < GM; ++h) {
    float x[NS];
    const bool live = h < grp;
    const __nv_bfloat16* src = q + ((int64_t)b * g.Hq + hkv * grp + (live ? h : 0)) * D + NS * lane;
#pragma unroll
    for (int i = 0; i < NS; ++i) x[i] = live ? __bfloat162float(src[i]) : 0.f;
    fwht_contig<D>(x, lane, inv_sqrt_d);
#pragma unroll
    for (int i = 0; i < NS; ++i) qr[h][i] = x[i] * c2;
  }
  float m[GM], l[GM], o[GM][NS];
#pragma unroll
  for (int h = 0; h < GM; ++h) {
    m[h] = -INFINITY;
    l[h] = 0.f;
#pragma unroll
    for (int i = 0; i < NS; ++i) o[h][i] = 0.f;
  }
  const int per = (te - ts + 7) / 8;
  const int w0 = ts + warp * per, w1 = min(te, w0 + per);
  const int kb = g.kb, vb = g.vb;
  const unsigned kmask = (1u << kb) - 1, vmask = (1u << vb) - 1;
  const int grpc = NS * lane / G;                   // this lane's channel group
  float qp[GM][NS], qs[GM];                         // q' = q_rot c_block and its lane sum
  float cv[NS];                                     // value column scales of the block
  int cur_blk = -1;
  for (int t = w0; t < w1; ++t) {
    float kv[NS], vv[NS];
    const bool coded = t >= S && t - S < nbq;
    float dot[GM];
    if (coded) {
      const int qi = t - S, blk = qi / G;
      if (blk != cur_blk) {                         // refold the block's column scales
        cur_blk = blk;
        const __half* ck = plane_ptr<__half>(g, KVQ_PLANE_K_COL, b, hkv, blk, NS * lane);
        const __half* cvp = plane_ptr<__half>(g, KVQ_PLANE_V_COL, b, hkv, blk, NS * lane);
#pragma unroll
        for (int i = 0; i < NS; ++i) {
          const float c = __half2float(ck[i]);
          cv[i] = __half2float(cvp[i]);
#pragma unroll
          for (int h = 0; h < GM; ++h) qp[h][i] = qr[h][i] * c;
        }
#pragma unroll
        for (int h = 0; h < GM; ++h) {
          float a = 0.f;
#pragma unroll
          for (int i = 0; i < NS; ++i) a += qp[h][i];
          qs[h] = a;
        }
      }
      const uint32_t wk = lane_codes(plane_ptr<uint8_t>(g, KVQ_PLANE_K_CODES, b, hkv, qi), lane, NS, kb);
      const uint32_t wv = lane_codes(plane_ptr<uint8_t>(g, KVQ_PLANE_V_CODES, b, hkv, qi), lane, NS, vb);
      const float ks = __half2float(*plane_ptr<__half>(g, KVQ_PLANE_K_SCALE, b, hkv, qi, grpc));
      const float kz = __half2float(*plane_ptr<__half>(g, KVQ_PLANE_K_ZERO, b, hkv, qi, grpc));
      const float kr = __half2float(*plane_ptr<__half>(g, KVQ_PLANE_K_ROW, b, hkv, 0, qi));
      const float vs = __half2float(*plane_ptr<__half>(g, KVQ_PLANE_V_SCALE, b, hkv, qi, grpc));
      const float vz = __half2float(*plane_ptr<__half>(g, KVQ_PLANE_V_ZERO, b, hkv, qi, grpc));
      const float vr = __half2float(*plane_ptr<__half>(g, KVQ_PLANE_V_ROW, b, hkv, 0, qi));
#pragma unroll
      for (int h = 0; h < GM; ++h) {
        float a = 0.f;
#pragma unroll
        for (int i = 0; i < NS; ++i) a += qp[h][i] * (float)((wk >> (i * kb)) & kmask);
        dot[h] = kr * (ks * a + kz * qs[h]);
      }
#pragma unroll
      for (int i = 0; i < NS; ++i) vv[i] = vr * cv[i] * ((float)((wv >> (i * vb)) & vmask) * vs + vz);
    } else {                                        // sink or staged: rotate forward
      const __nv_bfloat16* kp = t < S
          ? plane_ptr<__nv_bfloat16>(g, KVQ_PLANE_K_FULL, b, hkv, t, NS * lane)
          : plane_ptr<__nv_bfloat16>(g, KVQ_PLANE_K_PEND, b, hkv, (t - S) % G, NS * lane);
      const __nv_bfloat16* vp = t < S
          ? plane_ptr<__nv_bfloat16>(g, KVQ_PLANE_V_FULL, b, hkv, t, NS * lane)
          : plane_ptr<__nv_bfloat16>(g, KVQ_PLANE_V_PEND, b, hkv, (t - S) % G, NS * lane);
#pragma unroll
      for (int i = 0; i < NS; ++i) {
        kv[i] = __bfloat162float(kp[i]);
        vv[i] = __bfloat162float(vp[i]);
      }
      fwht_contig<D>(kv, lane, inv_sqrt_d);
      fwht_contig<D>(vv, lane, inv_sqrt_d);
#pragma unroll
      for (int h = 0; h < GM; ++h) {
        float a = 0.f;
#pragma unroll
        for (int i = 0; i < NS; ++i) a += qr[h][i] * kv[i];
        dot[h] = a;
      }
    }
#pragma unroll
    for (int h = 0; h < GM; ++h) {
      float sc = dot[h];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) sc += __shfl_xor_sync(0xffffffffu, sc, off);
      const float mn = fmaxf(m[h], sc);
      const float alpha = exp2f(m[h] - mn);         // m = -inf at first: alpha = 0
      const float p = exp2f(sc - mn);
      m[h] = mn;
      l[h] = l[h] * alpha + p;
#pragma unroll
      for (int i = 0; i < NS; ++i) o[h][i] = o[h][i] * alpha + p * vv[i];
    }
  }
  // ---- merge the warps, rotate back, write the split's partial ----
  float* red = ksm;                                  // [8][GM][D + 2]
#pragma unroll
  for (int h = 0; h < GM; ++h) {
    float* rw = red + (warp * GM + h) * (D + 2);
    if (lane == 0) {
      rw[0] = m[h];
      rw[1] = l[h];
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) rw[2 + NS * lane + i] = o[h][i];
  }
  __syncthreads();
  for (int h = warp; h < grp; h += 8) {
    float M = -INFINITY;
    for (int w = 0; w < 8; ++w) M = fmaxf(M, red[(w * GM + h) * (D + 2)]);
    float L = 0.f, x[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) x[i] = 0.f;
    for (int w = 0; w < 8; ++w) {
      const float* rw = red + (w * GM + h) * (D + 2);
      if (rw[0] == -INFINITY) continue;
      const float f = exp2f(rw[0] - M);
      L += f * rw[1];
#pragma unroll
      for (int i = 0; i < NS; ++i) x[i] += f * rw[2 + NS * lane + i];
    }
    fwht_contig<D>(x, lane, inv_sqrt_d);
    float* wsr = ws_row(g, b, hkv * grp + h) + (int64_t)split * (D + kWsStride);
    if (lane == 0) {
      wsr[0] = M == -INFINITY ? -INFINITY : M * 0.6931471805599453f;   // natural-log units
      wsr[1] = L;
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) wsr[2 + NS * lane + i] = x[i];
  }
  // ---- the last split CTA of this (sequence, kv head) merges the splits ----
  __shared__ int last_cta;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last_cta = atomicAdd(&g.counters[b * g.H + hkv], 1u) == (unsigned)g.splits - 1;
  }
  __syncthreads();
  if (!last_cta) return;
  __threadfence();
  const int n = g.splits;
  for (int h = warp; h < grp; h += 8) {
    const float* w = ws_row(g, b, hkv * grp + h);
    auto row = [&](int i) { return w + (int64_t)i * (D + kWsStride); };
    float M = -INFINITY;
    for (int i = lane; i < n; i += 32) M = fmaxf(M, __ldcg(row(i)));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
    float L = 0.f, acc[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) acc[i] = 0.f;
    for (int i = 0; i < n; ++i) {
      const float mi = __ldcg(row(i));
      if (mi == -INFINITY) continue;
      const float f = expf(mi - M);
      L += f * __ldcg(row(i) + 1);
#pragma unroll
      for (int k = 0; k < NS; ++k) acc[k] += f * __ldcg(row(i) + 2 + lane + 32 * k);
    }
#pragma unroll
    for (int k = 0; k < NS; ++k)
      st_act(out, ((int64_t)b * g.Hq + hkv * grp + h) * D + lane + 32 * k, acc[k] / L, g.act);
  }
  if (threadIdx.x == 0) g.counters[b * g.H + hkv] = 0;   // ready for the next call
}

template <int D>
cudaError_t launch_kvarn_d(const Geom& g, const void* q, float scale, void* out, cudaStream_t s) {
  const int grp = g.Hq / g.H;
  const float inv_sqrt_d = (float)(1.0 / sqrt((double)D));
  dim3 grid(g.splits, g.H, g.B);
  auto run = [&](auto kern, int gm) {
    const size_t sm = (size_t)8 * gm * (D + 2) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    launch_pdl(kern, dim3(grid), dim3(256), sm, s, g, reinterpret_cast<const __nv_bfloat16*>(q),
               scale, inv_sqrt_d, out);
    return cudaGetLastError();
  };
  if (grp <= 2) return run(attend_kvarn_decode_kernel<D, 2>, 2);
  if (grp <= 4) return run(attend_kvarn_decode_kernel<D, 4>, 4);
  return run(attend_kvarn_decode_kernel<D, 8>, 8);
}

bool kvarn_decode_supported(const Geom& g) {
  return g.fmt == KVQ_FMT_KVARN && g.act == KVQ_BF16 && (g.D == 64 || g.D == 128 || g.D == 256) &&
         g.Hq / g.H <= 8 && (g.kb == 2 || g.kb == 4) && (g.vb == 2 || g.vb == 4) &&
         g.G >= g.D / 32 && g.G % (g.D / 32) == 0;
}

}  // namespace

int decode_splits(const Geom& g) {
  // the split kernels fit two CTAs per SM: round down so that every split of
  // every (sequence, kv head) runs in the first wave
  const int bh = g.B * g.H;
  int s = 2 * num_sms() / bh;
  if (s > kMaxSplits - 1) s = kMaxSplits - 1;
  return s < 1 ? 1 : s;
}

cudaError_t launch_attend(const Geom& g, const void* q, int L, float scale, void* out,
                          bool decode, int t_hint, cudaStream_t s) {
  if (!decode && prefill_m256_supported(g)) {
    int* err = device_error_word();
    if (!err) return cudaErrorInvalidDevice;
    return launch_prefill_m256(g, q, L, scale, out, err, s);
  }
  // (short calls stay with the mma.sync kernel, whose time grows with tokens and queries
  // from 14 us on, where the tcgen05 pair takes 19-20 us to set up, rotate and store.  Four
  // sequences, 8 kv heads of 2 query heads, mma.sync / tcgen05: 16 tokens and queries
  // 17.4 / 19.7 us, 24 and 12 19.5 / 19.8, 32 and 4 18.6 / 19.9, 20 and 20 20.1 / 19.7,
  // 32 and 12 20.7 / 19.8)
  if (!decode && prefill_kvarn_supported(g) && t_hint + (int64_t)L > 36) {
    int* err = device_error_word();
    if (!err) return cudaErrorInvalidDevice;
    return launch_prefill_kvarn(g, q, L, scale, out, err, s);
  }
  if (!decode && prefill_mma_supported(g)) return launch_prefill_mma(g, q, L, scale, out, s);
  // the streaming decode pays off once every CTA streams a few stages; short
  // caches keep the split kernel (both read T on the device and are exact
  // for any T, so a captured graph stays correct as the cache grows)
  const int64_t blocks = (int64_t)g.B * g.H * ((t_hint + 31) / 32);
  if (decode && decode_stream_supported(g) &&
      (!decode_mma_supported(g) || blocks >= 16 * (int64_t)decode_stream_ctas(g))) {
    int* err = device_error_word();
    if (!err) return cudaErrorInvalidDevice;
    return launch_decode_stream(g, q, scale, err, out, s);
  }
  if (decode && decode_mma_supported(g)) {
    int* err = device_error_word();
    if (!err) return cudaErrorInvalidDevice;
    return launch_decode_mma(g, q, scale, err, out, s);
  }
  if (decode && kvarn_decode_supported(g)) {
    // long caches: the sinks and staged tokens leave partials, then the coded
    // tokens go through the tensor cores and everything is merged
    const int64_t coded = (int64_t)g.B * g.H * (kvarn_nblocks(t_hint, g.S, g.G) * g.G / 32);
    if (decode_stream_kvarn_supported(g) && coded >= 16 * (int64_t)decode_stream_ctas(g)) {
      int* err = device_error_word();
      if (!err) return cudaErrorInvalidDevice;
      return launch_decode_stream_kvarn(g, q, scale, err, out, s);
    }
    return g.D == 64 ? launch_kvarn_d<64>(g, q, scale, out, s)
         : g.D == 128 ? launch_kvarn_d<128>(g, q, scale, out, s)
                      : launch_kvarn_d<256>(g, q, scale, out, s);
  }
  return g.D == 64 ? launch_generic_d<64>(g, q, L, scale, out, decode, s)
       : g.D == 128 ? launch_generic_d<128>(g, q, L, scale, out, decode, s)
                    : launch_generic_d<256>(g, q, L, scale, out, decode, s);
}

}  // namespace kvq
