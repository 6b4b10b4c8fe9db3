// Streaming decode attention over the coded tokens of a KVarN cache, on
// tensor cores in the Hadamard-rotated basis (§3.1 KVarN: coded token t is
// stored as r_t c_j (s_tg code_tj + m_tg) with row scale r_t, per-block column
// scale c_j and per-token group scale/offset; §3.2-3.3 attention over the
// stored reconstruction, L = 1).
//
// The work split, the ring and the merges follow decode_stream.cu: persistent
// CTAs stream equal shares of the flattened (sequence, kv head, 32-token
// block) space of coded blocks; a producer warp copies runs of blocks (codes,
// group metadata, row scales) and each block's column-scale rows into ring
// stages; eleven consumer warps take the blocks in turn, tokens as the MMA rows
// and the GQA heads as its columns.
//   scores  q_rot = H q / sqrt(D) (times the softmax scale in log2 units) is
//     formed once per head; per block B = q_rot * c_k as bf16 high + low parts
//     and A = key codes as exact bf16 integers 128 + c, one accumulator per
//     quantization group; the 128 is removed with an MMA over a constant
//     operand (which also gives sum_j q'_j, the offset's weight), then
//       S = r_t sum_g [s_tg (acc_g - bias_g) + m_tg bias_g / 128].
//   values  A = codes read in place as exact subnormal fp16, B = fp16(p) *
//     (r_t s_tg), one accumulator set per block and group; c_v,j is applied when the
//     block's sums are added, with the offsets r_t m_tg from a small MMA (rows =
//     groups).
// The sinks and the staged tokens (full precision, original basis: no rotation
// is needed to attend them) go through kvarn_full_kernel, launched first: four
// CTAs per head, a warp per token, partials in the top workspace slots.  The
// streaming kernel starts while it runs (programmatic launch) and waits for it
// only where it merges: the head's last CTA rotates the coded tokens' output back
// and adds the four partials.  12B-class shape, batch 4, 8300 tokens: the split kernel
// that used to take the full-precision tokens after the streaming kernel, rotating
// each of them, added 17 us to its 52 (four layers: 274 -> 241 us).
#include <type_traits>

#include "decode_attn.cuh"
#include "ring_pass.h"
#include "stream_common.cuh"

namespace kvq {
namespace {
using namespace dattn;
using namespace stream;

template <int D, int KB, int VB, int G>
struct KCfg {
  static constexpr int NG32 = D / 32;                 // 32-channel sub-groups (two k-steps each)
  static constexpr int NGG = D / G;                   // quantization groups per token
  static constexpr int MT = D / 16;                   // P V m-tiles
  static constexpr int KCB = D * KB / 8, VCB = D * VB / 8;
  static constexpr int MB = kBT * NGG * 2;            // one group-metadata plane of a block
  // a stage holds kSB consecutive blocks; each plane is contiguous over them
  static constexpr int KC = 0;
  static constexpr int VC = KC + kSB * kBT * KCB;
  static constexpr int KS = VC + kSB * kBT * VCB;
  static constexpr int KZ = KS + kSB * MB;
  static constexpr int VS = KZ + kSB * MB;
  static constexpr int VZ = VS + kSB * MB;
  static constexpr int KR = VZ + kSB * MB;            // row scales, 2 bytes per token
  static constexpr int VR = KR + kSB * kBT * 2;
  static constexpr int KCOL = VR + kSB * kBT * 2;     // one column-scale row per block
  static constexpr int VCOL = KCOL + kSB * D * 2;
  static constexpr int STAGE = (VCOL + kSB * D * 2 + 127) / 128 * 128;
  static_assert(G % kBT == 0 && G % 32 == 0, "blocks lie inside one column-scale block");
  static_assert(NGG <= 8, "offset MMA rows hold the groups");
};

// The MMAs without `volatile`: the compiler may move them among independent ones.
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                        uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Normalised Hadamard transform of a row held as x[i] = row[lane + 32 i]
// (butterflies over the lanes, then over the slots, then 1 / sqrt(D)).
template <int D>
__device__ __forceinline__ void fwht_rows(float (&x)[D / 32], int lane, float inv_sqrt_d) {
  constexpr int NS = D / 32;
#pragma unroll
  for (int h = 1; h < 32; h <<= 1)
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      const float y = __shfl_xor_sync(0xffffffffu, x[i], h);
      x[i] = (lane & h) ? y - x[i] : x[i] + y;
    }
#pragma unroll
  for (int hs = 1; hs < NS; hs <<= 1)
#pragma unroll
    for (int i = 0; i < NS; ++i)
      if (!(i & hs)) {
        const float a = x[i], c = x[i + hs];
        x[i] = a + c;
        x[i + hs] = a - c;
      }
#pragma unroll
  for (int i = 0; i < NS; ++i) x[i] *= inv_sqrt_d;
}

// Attention of every query head of one (sequence, kv head) over one of
// kFullSplits shares of its full-precision tokens.  Lane l holds channels
// NS l .. of the queries; a warp takes four tokens at a time, so that eight row
// loads are in flight.  Partials (m in log2 units, l, o) go to workspace slots
// kFullSlot ...
constexpr int kFullWarps = 4;

template <int D, int GM>
__global__ void __launch_bounds__(kFullWarps * 32)
kvarn_full_kernel(Geom g, const __nv_bfloat16* __restrict__ q, float scale) {
  pdl_wait();
  pdl_trigger();
  constexpr int NS = D / 32, NB = 4;
  __shared__ float red[kFullWarps][GM][D + 2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int hkv = blockIdx.y, b = blockIdx.z, grp = g.Hq / g.H, S = g.S;
  const int T = cache_tokens(g);
  const int nbq = kvarn_nblocks(T, S, g.G) * g.G;
  const int per = (T - nbq + kFullSplits - 1) / kFullSplits;
  const int ts = blockIdx.x * per, te = min(T - nbq, ts + per);
  const float c2 = scale * 1.4426950408889634f;   // scores in log2 units
  struct __align__(NS * 2) Row { __nv_bfloat162 v[NS / 2]; };
  float qf[GM][NS], o[GM][NS], m[GM], l[GM];
#pragma unroll
  for (int h = 0; h < GM; ++h) {
    m[h] = -INFINITY;
    l[h] = 0.f;
    Row r = {};
    if (h < grp)
      r = *reinterpret_cast<const Row*>(q + ((int64_t)b * g.Hq + hkv * grp + h) * D + NS * lane);
#pragma unroll
    for (int i = 0; i < NS / 2; ++i) {
      const float2 f = __bfloat1622float2(r.v[i]);
      qf[h][2 * i] = f.x * c2;
      qf[h][2 * i + 1] = f.y * c2;
      o[h][2 * i] = o[h][2 * i + 1] = 0.f;
    }
  }
  for (int f0 = ts + warp * NB; f0 < te; f0 += kFullWarps * NB) {
    Row kr[NB], vr[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int f = min(f0 + u, te - 1);          // sinks, then staged tokens
      const int slot = f < S ? f : (f + nbq - S) % g.G;
      kr[u] = *reinterpret_cast<const Row*>(plane_ptr<__nv_bfloat16>(
          g, f < S ? KVQ_PLANE_K_FULL : KVQ_PLANE_K_PEND, b, hkv, slot, NS * lane));
      vr[u] = *reinterpret_cast<const Row*>(plane_ptr<__nv_bfloat16>(
          g, f < S ? KVQ_PLANE_V_FULL : KVQ_PLANE_V_PEND, b, hkv, slot, NS * lane));
    }
    float sc[GM][NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      float kf[NS];
#pragma unroll
      for (int i = 0; i < NS / 2; ++i) {
        const float2 f = __bfloat1622float2(kr[u].v[i]);
        kf[2 * i] = f.x;
        kf[2 * i + 1] = f.y;
      }
#pragma unroll
      for (int h = 0; h < GM; ++h) {
        float d = 0.f;
#pragma unroll
        for (int i = 0; i < NS; ++i) d = fmaf(qf[h][i], kf[i], d);
        sc[h][u] = d;
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
      for (int h = 0; h < GM; ++h)
#pragma unroll
        for (int u = 0; u < NB; ++u) sc[h][u] += __shfl_xor_sync(0xffffffffu, sc[h][u], off);
#pragma unroll
    for (int h = 0; h < GM; ++h) {
      float mn = m[h];
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        if (f0 + u >= te) sc[h][u] = -INFINITY;
        mn = fmaxf(mn, sc[h][u]);
      }
      const float alpha = exp2f(m[h] - mn);       // m = -inf at first: 0
      m[h] = mn;
      l[h] *= alpha;
#pragma unroll
      for (int i = 0; i < NS; ++i) o[h][i] *= alpha;
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        sc[h][u] = exp2f(sc[h][u] - mn);
        l[h] += sc[h][u];
      }
    }
#pragma unroll
    for (int u = 0; u < NB; ++u)
#pragma unroll
      for (int i = 0; i < NS / 2; ++i) {
        const float2 f = __bfloat1622float2(vr[u].v[i]);
#pragma unroll
        for (int h = 0; h < GM; ++h) {
          o[h][2 * i] = fmaf(sc[h][u], f.x, o[h][2 * i]);
          o[h][2 * i + 1] = fmaf(sc[h][u], f.y, o[h][2 * i + 1]);
        }
      }
  }
#pragma unroll
  for (int h = 0; h < GM; ++h) {
    if (lane == 0) {
      red[warp][h][0] = m[h];
      red[warp][h][1] = l[h];
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) red[warp][h][2 + NS * lane + i] = o[h][i];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < grp * (D + 2); i += kFullWarps * 32) {
    const int h = i / (D + 2), c = i % (D + 2);
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < kFullWarps; ++w) M = fmaxf(M, red[w][h][0]);
    float x = M;
    if (c > 0) {
      x = 0.f;
#pragma unroll
      for (int w = 0; w < kFullWarps; ++w)
        if (red[w][h][0] != -INFINITY) x += exp2f(red[w][h][0] - M) * red[w][h][c];
    }
    reinterpret_cast<float*>(g.pl[KVQ_PLANE_WORKSPACE].p)[
        (((int64_t)b * g.Hq + hkv * grp + h) * kMaxSplits + kFullSlot + blockIdx.x) * (D + kWsStride) + c] = x;
  }
}

// One head's output: the coded tokens' rotated-back row x[i] = channel lane + 32 i
// (m in log2 units and l; -inf and 0 if there are none) and the
// full-precision tokens' partials wf (the head's workspace slot kFullSlot ...).
template <int D>
__device__ __forceinline__ void merge_full(const float* wf, float (&x)[D / 32], float m, float l,
                                           int lane, __nv_bfloat16* out) {
  constexpr int R = D + kWsStride;
  float mf[kFullSplits], M = m;
#pragma unroll
  for (int s = 0; s < kFullSplits; ++s) {
    mf[s] = __ldcg(wf + s * R);
    M = fmaxf(M, mf[s]);
  }
  const float fx = m == -INFINITY ? 0.f : exp2f(m - M);
  float L = fx * l;
#pragma unroll
  for (int i = 0; i < D / 32; ++i) x[i] = m == -INFINITY ? 0.f : x[i] * fx;
#pragma unroll
  for (int s = 0; s < kFullSplits; ++s) {
    if (mf[s] == -INFINITY) continue;
    const float f = exp2f(mf[s] - M);
    L = fmaf(f, __ldcg(wf + s * R + 1), L);
#pragma unroll
    for (int i = 0; i < D / 32; ++i) x[i] = fmaf(f, __ldcg(wf + s * R + 2 + lane + 32 * i), x[i]);
  }
#pragma unroll
  for (int i = 0; i < D / 32; ++i) out[lane + 32 * i] = __float2bfloat16_rn(x[i] / L);
}

// Floats of the warps' partials of `pw` floats each, up to the next 16 bytes: the
// queries behind them are read four at a time, and pw is not a multiple of four
// where the group is odd.
__host__ __device__ constexpr int slot_floats(int pw) { return (kNW * pw + 3) / 4 * 4; }

// Launched after kvarn_full_kernel, whose start waited for everything before it:
// only its partials have to be waited for (pdl_wait before the merges).
// PAIR: at most two query heads per kv head.
template <int D, int KB, int VB, int G, bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
decode_stream_kvarn_kernel(Geom g, const __nv_bfloat16* __restrict__ q, float scale,
                           float inv_sqrt_d, int* err, __nv_bfloat16* __restrict__ out, int ns) {
  static_assert(KB == 4 && VB == 2, "the code layouts below");
  using C = KCfg<D, KB, VB, G>;
  constexpr int NG32 = C::NG32, NGG = C::NGG, MT = C::MT;
  constexpr int CPL = G / 8;                         // channels of a group per value row (gid)
  constexpr int GT = CPL / 2;                        // P V m-tiles per group
  extern __shared__ __align__(128) unsigned char smem[];
  pdl_trigger();

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gid = lane >> 2, tid = lane & 3;
  const int grp = g.Hq / g.H;
  const int PW = grp * (D + 2);
  float* slot = reinterpret_cast<float*>(smem + (size_t)ns * C::STAGE);   // [kNW][PW]
  float* qr = slot + slot_floats(PW);                // [8][D] rotated queries, then merged rows
  Merge* mg = reinterpret_cast<Merge*>(qr + 8 * D);
  uint64_t* full = reinterpret_cast<uint64_t*>(mg + 1);
  uint64_t* empty = full + ns;
  float* wsb = reinterpret_cast<float*>(g.pl[KVQ_PLANE_WORKSPACE].p);

  const int T = cache_tokens(g);
  const int S = g.S;
  const int nbq = kvarn_nblocks(T, S, G) * G;        // coded tokens per head
  const int BH = g.B * g.H;
  const int nb = nbq / kBT;                          // blocks per head
  const int64_t N = (int64_t)BH * nb;
  if (N == 0) {                                      // nothing coded
    pdl_wait();
    for (int i = blockIdx.x * (kThreads / 32) + warp; i < g.B * g.Hq; i += gridDim.x * (kThreads / 32)) {
      float x[D / 32];
      merge_full<D>(wsb + ((int64_t)i * kMaxSplits + kFullSlot) * (D + kWsStride), x, -INFINITY, 0.f,
                    lane, out + (int64_t)i * D);
    }
    return;
  }
  const int P = N < (int64_t)gridDim.x ? (int)N : (int)gridDim.x;
  if ((int)blockIdx.x >= P) return;
  const int64_t k0 = range_start(blockIdx.x, N, P), k1 = range_start(blockIdx.x + 1, N, P);
  const int nblk = (int)(k1 - k0);

  if (threadIdx.x == 0) {
    for (int i = 0; i < ns; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kNW);                     // every consumer warp leaves every stage
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  // ------------------------------------------------------------------ producer
  if (warp == kNW) {
    const int nst = (nblk + kSB - 1) / kSB;
    int head = (int)(k0 / nb), blk = (int)(k0 % nb);  // first block of the next stage
    int s = 0;
    for (; s < nst; ++s) {
      const int st = s % ns;
      bool ok = true;
      if (s >= ns && lane == 0) ok = mbar_wait(&empty[st], ((s / ns) - 1) & 1);
      if (!__shfl_sync(0xffffffffu, ok, 0)) {
        if (lane == 0) atomicOr(err, 1);
        break;
      }
      const int nbs = min(kSB, nblk - s * kSB);
      const int h_st = head, b_st = blk;
      unsigned char* sp = smem + (size_t)st * C::STAGE;
      if (lane == 0)
        mbar_expect_tx(&full[st], (uint32_t)nbs * (kBT * (C::KCB + C::VCB) + 4 * C::MB +
                                                   2 * kBT * 2 + 2 * D * 2));
      __syncwarp();
      // runs of one head's blocks: in pass p, lane 8 r + c issues copy c of
      // run 4 p + r (every lane walks the same blocks)
      int nrun = 0;
      for (int pass = 0; pass == 0 || pass * 4 < nrun; ++pass) {
        const int myr = pass * 4 + lane / 8, myc = lane % 8;
        int hh = h_st, bb = b_st, cnt = 0, r_head = 0, r_blk = 0, r_n = 0, r_sub = 0, p_head = -1;
#pragma unroll
        for (int i = 0; i < kSB; ++i) {
          if (i < nbs) {
            if (hh != p_head) {
              if (cnt == myr) { r_head = hh; r_blk = bb; r_sub = i; }
              ++cnt;
              p_head = hh;
            }
            if (cnt - 1 == myr) ++r_n;
            if (++bb == nb) { bb = 0; ++hh; }
          }
        }
        if (pass == 0) {
          nrun = cnt;
          head = hh;
          blk = bb;
        }
        if (myr < nrun) {
          const int qi = r_blk * kBT, nt = r_n * kBT;   // coded-token rows of the run
          const uint8_t* src;
          unsigned char* dst;
          uint32_t bytes;
          const int planes[8] = {KVQ_PLANE_K_CODES, KVQ_PLANE_V_CODES, KVQ_PLANE_K_SCALE,
                                 KVQ_PLANE_K_ZERO, KVQ_PLANE_V_SCALE, KVQ_PLANE_V_ZERO,
                                 KVQ_PLANE_K_ROW, KVQ_PLANE_V_ROW};
          if (myc < 2) {
            src = plane_ptr<uint8_t>(g, planes[myc], 0, r_head, qi);
            dst = sp + (myc == 0 ? C::KC + r_sub * kBT * C::KCB : C::VC + r_sub * kBT * C::VCB);
            bytes = nt * (myc == 0 ? C::KCB : C::VCB);
          } else if (myc < 6) {
            src = reinterpret_cast<const uint8_t*>(plane_ptr<__half>(g, planes[myc], 0, r_head, qi));
            dst = sp + C::KS + (myc - 2) * kSB * C::MB + r_sub * C::MB;
            bytes = r_n * C::MB;
          } else {                                     // row scales: plane row 0, column qi
            src = reinterpret_cast<const uint8_t*>(plane_ptr<__half>(g, planes[myc], 0, r_head, 0, qi));
            dst = sp + (myc == 6 ? C::KR : C::VR) + r_sub * kBT * 2;
            bytes = nt * 2;
          }
          bulk_g2s(dst, src, bytes, &full[st]);
        }
      }
      // each block's column-scale rows (key, value)
      if (lane < 2 * nbs) {
        const int i = lane >> 1, which = lane & 1;
        int hh = h_st, bb = b_st;
#pragma unroll
        for (int j = 0; j < kSB; ++j)
          if (j < i && ++bb == nb) { bb = 0; ++hh; }
        const int crow = bb * kBT / G;
        bulk_g2s(sp + (which ? C::VCOL : C::KCOL) + i * D * 2,
                 plane_ptr<__half>(g, which ? KVQ_PLANE_V_COL : KVQ_PLANE_K_COL, 0, hh, crow),
                 D * 2, &full[st]);
      }
    }
    if (lane == 0)                                   // the last copies land before the CTA ends
      for (int i = max(0, s - ns); i < s; ++i)
        if (!mbar_wait(&full[i % ns], (i / ns) & 1)) atomicOr(err, 1);
    return;
  }

  // ------------------------------------------------------------------ consumers
  const float c2 = scale * 1.4426950408889634f;      // scores in log2 units
  constexpr uint32_t kmask = 0x000F000Fu;
  const uint32_t a128[4] = {kMagic, kMagic, kMagic, kMagic};
  const int tc = threadIdx.x;

  float m_run[2], l_run[2];
  float o[MT][4];
  bool bad = false;
  static_assert(kSB <= kNW, "a warp has one block of a stage at most");
  int next = 0;                                      // first stage this warp (lane 0) has not left
  auto wait_stage = [&](int s) { return mbar_wait(&full[s % ns], (s / ns) & 1); };
  auto leave_stage = [&](int s) { mbar_arrive1(&empty[s % ns]); };

  auto process = [&](const unsigned char* sp, int sub) {
    const unsigned char* kc = sp + C::KC + sub * kBT * C::KCB;
    const unsigned char* vc = sp + C::VC + sub * kBT * C::VCB;
    const __half* ks = reinterpret_cast<const __half*>(sp + C::KS + sub * C::MB);
    const __half* kz = reinterpret_cast<const __half*>(sp + C::KZ + sub * C::MB);
    const uint32_t* vs = reinterpret_cast<const uint32_t*>(sp + C::VS + sub * C::MB);
    const uint32_t* vz = reinterpret_cast<const uint32_t*>(sp + C::VZ + sub * C::MB);
    const __half* kr = reinterpret_cast<const __half*>(sp + C::KR + sub * kBT * 2);
    const uint16_t* vr = reinterpret_cast<const uint16_t*>(sp + C::VR + sub * kBT * 2);
    const __half* kcol = reinterpret_cast<const __half*>(sp + C::KCOL + sub * D * 2);
    const __half* vcol = reinterpret_cast<const __half*>(sp + C::VCOL + sub * D * 2);

    // ---------------------------------------------------------------- scores
    // One group at a time: its G / 32 words per lane (8 codes each) of channels
    // G gg + G / 4 tid + 8 w, then its share of the scores.
    using GroupHalves = typename std::conditional<NGG == 4, uint2, uint32_t>::type;   // NGG fp16 of a token
    static_assert(NGG * 2 == sizeof(GroupHalves), "a token's group metadata in one load");
    GroupHalves ksv[4], kzv[4];
    float S[2][4] = {};
#pragma unroll
    for (int i = 0; i < 4; ++i) {                    // tokens gid + 8 i
      ksv[i] = *reinterpret_cast<const GroupHalves*>(ks + (gid + 8 * i) * NGG);
      kzv[i] = *reinterpret_cast<const GroupHalves*>(kz + (gid + 8 * i) * NGG);
    }
    uint32_t qh[4], ql[4];                           // q' of one word: [sb][half] high, low parts
    auto fold = [&](int head, int unit, uint32_t (&h4)[4], uint32_t (&l4)[4]) {
      // q' = q_rot * c_k of the word's 8 channels, as bf16 high and low parts
      const int ch = unit * 32 / G * G + (G / 4) * tid + 8 * (unit % (G / 32));
      const float4 qa = *reinterpret_cast<const float4*>(qr + head * D + ch);
      const float4 qb4 = *reinterpret_cast<const float4*>(qr + head * D + ch + 4);
      const uint4 cu = *reinterpret_cast<const uint4*>(kcol + ch);
      const __half2* c2p = reinterpret_cast<const __half2*>(&cu);
      float x[8] = {qa.x, qa.y, qa.z, qa.w, qb4.x, qb4.y, qb4.z, qb4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 cf = __half22float2(c2p[e]);
        x[2 * e] *= cf.x;
        x[2 * e + 1] *= cf.y;
      }
#pragma unroll
      for (int sb = 0; sb < 2; ++sb)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const int e0 = qk_chan<KB>(sb, hf, 0), e1 = qk_chan<KB>(sb, hf, 1);
          const uint32_t hw = pack_bf16(x[e0], x[e1]);
          const float2 hv = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hw));
          h4[2 * sb + hf] = hw;
          l4[2 * sb + hf] = pack_bf16(x[e0] - hv.x, x[e1] - hv.y);
        }
    };
    uint32_t sh[4], sl[4];                           // q' that this lane forms for the others
#pragma unroll
    for (int gg = 0; gg < NGG; ++gg) {
      float acc[2][4] = {}, bias[4] = {};
      uint32_t kw[4][G / 32];
#pragma unroll
      for (int i = 0; i < 4; ++i) {                  // rows gid + 8 i
        const unsigned char* r = kc + (gid + 8 * i) * C::KCB + gg * (G / 2) + tid * (G / 8);
        if constexpr (G == 64) {
          const uint2 u = *reinterpret_cast<const uint2*>(r);
          kw[i][0] = u.x;
          kw[i][1] = u.y;
        } else {
          kw[i][0] = *reinterpret_cast<const uint32_t*>(r);
        }
      }
#pragma unroll
      for (int w = 0; w < G / 32; ++w) {
        const int unit = gg * (G / 32) + w;
        if (PAIR) {
          // two heads at most: the eight lanes that share a tid form two words
          // of q' in turn (head gid % 2, word gid / 2) and pass them on; the
          // columns beyond the group repeat the two heads and are not stored
          constexpr int RND = NG32 < 4 ? NG32 : 4;
          if (unit % RND == 0) fold(gid & 1, unit + (gid >> 1) % RND, sh, sl);
          const int src = ((unit % RND) * 2 + (gid & 1)) * 4 + tid;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            qh[i] = __shfl_sync(0xffffffffu, sh[i], src);
            ql[i] = __shfl_sync(0xffffffffu, sl[i], src);
          }
        } else {
          fold(gid, unit, qh, ql);
        }
#pragma unroll
        for (int sb = 0; sb < 2; ++sb) {
          uint32_t a[2][4];
#pragma unroll
          for (int mt = 0; mt < 2; ++mt) {
            const uint32_t w0 = kw[2 * mt][w], w1 = kw[2 * mt + 1][w];
            a[mt][0] = magic2(w0 >> (8 * sb), kmask);
            a[mt][1] = magic2(w1 >> (8 * sb), kmask);
            a[mt][2] = magic2(w0 >> (8 * sb + 4), kmask);
            a[mt][3] = magic2(w1 >> (8 * sb + 4), kmask);
          }
          // (in an order that keeps MMAs on one accumulator apart)
          mma_bf16(bias, a128, qh[2 * sb], qh[2 * sb + 1]);
          mma_bf16(acc[0], a[0], qh[2 * sb], qh[2 * sb + 1]);
          mma_bf16(acc[1], a[1], qh[2 * sb], qh[2 * sb + 1]);
          mma_bf16(bias, a128, ql[2 * sb], ql[2 * sb + 1]);
          mma_bf16(acc[0], a[0], ql[2 * sb], ql[2 * sb + 1]);
          mma_bf16(acc[1], a[1], ql[2 * sb], ql[2 * sb + 1]);
        }
      }
      const float bz0 = bias[0] * (1.f / 128.f), bz1 = bias[1] * (1.f / 128.f);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float sc = __half2float(reinterpret_cast<const __half*>(&ksv[i])[gg]);
        const float mz = __half2float(reinterpret_cast<const __half*>(&kzv[i])[gg]);
        float* Si = &S[i >> 1][2 * (i & 1)];
        const float* ai = &acc[i >> 1][2 * (i & 1)];
        Si[0] += sc * (ai[0] - bias[0]) + mz * bz0;
        Si[1] += sc * (ai[1] - bias[1]) + mz * bz1;
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float rt = __half2float(kr[gid + 8 * i]);
      S[i >> 1][2 * (i & 1)] *= rt;
      S[i >> 1][2 * (i & 1) + 1] *= rt;
    }

    // --------------------------------------------------------------- softmax
    float mx[2];
#pragma unroll
    for (int jh = 0; jh < 2; ++jh) {
      mx[jh] = fmaxf(fmaxf(S[0][jh], S[0][2 + jh]), fmaxf(S[1][jh], S[1][2 + jh]));
      mx[jh] = fmaxf(mx[jh], __shfl_xor_sync(0xffffffffu, mx[jh], 4));
      mx[jh] = fmaxf(mx[jh], __shfl_xor_sync(0xffffffffu, mx[jh], 8));
      mx[jh] = fmaxf(mx[jh], __shfl_xor_sync(0xffffffffu, mx[jh], 16));
    }
    float alpha[2];
#pragma unroll
    for (int jh = 0; jh < 2; ++jh) {
      const float mn = fmaxf(m_run[jh], mx[jh]);
      alpha[jh] = m_run[jh] == -INFINITY ? 0.f : exp2f(m_run[jh] - mn);
      m_run[jh] = mn;
      l_run[jh] *= alpha[jh];
    }
    if (__any_sync(0xffffffffu, alpha[0] != 1.f || alpha[1] != 1.f)) {
#pragma unroll
      for (int i = 0; i < MT; ++i) {
        o[i][0] *= alpha[0]; o[i][1] *= alpha[1];
        o[i][2] *= alpha[0]; o[i][3] *= alpha[1];
      }
    }
    uint32_t pb[2][2];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      float p[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        p[i] = exp2f(S[mt][i] - m_run[i & 1]);
        l_run[i & 1] += p[i];
      }
      pb[mt][0] = movmatrix_t(pack_f16(p[0], p[1]));
      pb[mt][1] = movmatrix_t(pack_f16(p[2], p[3]));
    }

    // ------------------------------------------------------------------- P V
    // Value codes are read in place: bits 2 j, 2 j + 1 of a half word, masked,
    // are the code times 2^(2 j) as a subnormal fp16 (times 2^-24), exact in the
    // product; 2^(24 - 2 j) and the column scale are applied once per block in fp32.
    float offb[4] = {0.f, 0.f, 0.f, 0.f};            // sum_t p r_t m_tg, rows = groups
    uint32_t bq[NGG][2][2];                          // B = P (r_t s_tg) per group
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      const int t0 = 16 * mt + 2 * tid;              // tokens t0, t0 + 1 and t0 + 8, t0 + 9
      const uint32_t vr01 = *reinterpret_cast<const uint32_t*>(vr + t0);
      const uint32_t vr89 = *reinterpret_cast<const uint32_t*>(vr + t0 + 8);
      uint32_t a_off[4] = {0u, 0u, 0u, 0u};
      if (gid < NGG) {
        const uint16_t* vzh = reinterpret_cast<const uint16_t*>(vz) + t0 * NGG + gid;
        a_off[0] = hmul2u(vr01, (uint32_t)vzh[0] | ((uint32_t)vzh[NGG] << 16));
        a_off[2] = hmul2u(vr89, (uint32_t)vzh[8 * NGG] | ((uint32_t)vzh[9 * NGG] << 16));
      }
      mma_f16(offb, a_off, pb[mt][0], pb[mt][1]);
      const uint16_t* vsh = reinterpret_cast<const uint16_t*>(vs) + t0 * NGG;
      GroupHalves sv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        sv[i] = *reinterpret_cast<const GroupHalves*>(vsh + ((i & 1) + 8 * (i >> 1)) * NGG);
#pragma unroll
      for (int gg = 0; gg < NGG; ++gg) {
        const uint32_t sel = gg & 1 ? 0x7632 : 0x5410;
        const uint32_t s01 = __byte_perm(reinterpret_cast<const uint32_t*>(&sv[0])[gg >> 1],
                                         reinterpret_cast<const uint32_t*>(&sv[1])[gg >> 1], sel);
        const uint32_t s89 = __byte_perm(reinterpret_cast<const uint32_t*>(&sv[2])[gg >> 1],
                                         reinterpret_cast<const uint32_t*>(&sv[3])[gg >> 1], sel);
        bq[gg][mt][0] = hmul2u(pb[mt][0], hmul2u(vr01, s01));
        bq[gg][mt][1] = hmul2u(pb[mt][1], hmul2u(vr89, s89));
      }
    }
#pragma unroll
    for (int gg = 0; gg < NGG; ++gg) {
      float blk[GT][4] = {};                         // tile i: channels G gg + CPL gid + 2 i, + 1
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        // the lane's CPL channels of four tokens
        const unsigned char* v0 = vc + (16 * mt + 2 * tid) * C::VCB + gg * (G / 4) + gid * (CPL / 4);
        uint32_t x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const unsigned char* vp = v0 + ((i & 1) + 8 * (i >> 1)) * C::VCB;
          x[i] = CPL == 8 ? *reinterpret_cast<const uint16_t*>(vp) : *vp;
        }
        uint32_t x01 = x[0] | (x[1] << 16), x89 = x[2] | (x[3] << 16);
#pragma unroll
        for (int i = 0; i < GT; ++i) {
          if (i == 2) {                              // the upper byte of each half word
            x01 >>= 8;
            x89 >>= 8;
          }
          const uint32_t m0 = 0x00030003u << (4 * (i & 1)), m1 = m0 << 2;
          const uint32_t a[4] = {x01 & m0, x01 & m1, x89 & m0, x89 & m1};
          mma_f16(blk[i], a, bq[gg][mt][0], bq[gg][mt][1]);
        }
      }
      const float f0 = __shfl_sync(0xffffffffu, offb[0], 4 * gg + tid);
      const float f1 = __shfl_sync(0xffffffffu, offb[1], 4 * gg + tid);
      const __half2* cc = reinterpret_cast<const __half2*>(vcol + G * gg + CPL * gid);
#pragma unroll
      for (int i = 0; i < GT; ++i) {
        const float2 c = __half22float2(cc[i]);
        const float e0 = (float)(1 << (24 - 4 * (i & 1))), e1 = e0 * 0.25f;
        float* oi = o[GT * gg + i];
        oi[0] = fmaf(c.x, fmaf(blk[i][0], e0, f0), oi[0]);
        oi[1] = fmaf(c.x, fmaf(blk[i][1], e0, f1), oi[1]);
        oi[2] = fmaf(c.y, fmaf(blk[i][2], e1, f0), oi[2]);
        oi[3] = fmaf(c.y, fmaf(blk[i][3], e1, f1), oi[3]);
      }
    }
  };

  // the output of head rows h < grp from merged rows in qr (m in log2 units,
  // rotated o): rotate back, add the full-precision tokens' partials
  auto finish = [&](int b, int hkv, const float* Mh, const float* Lh) {
    consumer_sync();
    pdl_wait();
    if (warp < grp) {
      float x[D / 32];
#pragma unroll
      for (int i = 0; i < D / 32; ++i) x[i] = qr[warp * D + lane + 32 * i];
      fwht_rows<D>(x, lane, inv_sqrt_d);
      const int64_t row = (int64_t)b * g.Hq + hkv * grp + warp;
      merge_full<D>(wsb + (row * kMaxSplits + kFullSlot) * (D + kWsStride), x, Mh[warp], Lh[warp], lane,
                    out + row * D);
    }
    consumer_sync();
  };

  const int hfirst = (int)(k0 / nb), hlast = (int)((k1 - 1) / nb);
  for (int hd = hfirst; hd <= hlast; ++hd) {
    const int64_t hs = (int64_t)hd * nb;
    const int a = (int)(max(k0, hs) - k0), e = (int)(min(k1, hs + nb) - k0);
    const int b = hd / g.H, hkv = hd % g.H;
    // rotated queries of the head (times the softmax scale, log2 units):
    // rows 0-7 of qr, zero for the MMA columns beyond the group
    if (warp < 8) {
      float x[D / 32];
      const bool live = warp < grp;
      const __nv_bfloat16* src = q + ((int64_t)b * g.Hq + hkv * grp + (live ? warp : 0)) * D;
#pragma unroll
      for (int i = 0; i < D / 32; ++i) x[i] = live ? __bfloat162float(src[lane + 32 * i]) : 0.f;
      fwht_rows<D>(x, lane, inv_sqrt_d);
#pragma unroll
      for (int i = 0; i < D / 32; ++i) qr[warp * D + lane + 32 * i] = x[i] * c2;
    }
    consumer_sync();
    const int jst = a + ((warp - a) % kNW + kNW) % kNW;
    const bool mine = jst < e;
    m_run[0] = m_run[1] = -INFINITY;
    l_run[0] = l_run[1] = 0.f;
#pragma unroll
    for (int i = 0; i < MT; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
    for (int j = jst; j < e && !bad; j += kNW) {
      const int sj = j / kSB, st = sj % ns;
      bool ok = true;
      if (lane == 0) ok = ring_pass(next, sj, wait_stage, leave_stage) && wait_stage(sj);
      if (!__shfl_sync(0xffffffffu, ok, 0)) {
        if (lane == 0) atomicOr(err, 1);
        bad = true;
        break;
      }
      process(smem + (size_t)st * C::STAGE, j % kSB);
      __syncwarp();
      if (lane == 0) leave_stage(next++);
    }
    // the other warps may still be waiting for stages of this head: leave all that
    // come before its last one (which can hold a block of the next head for this warp)
    if (lane == 0 && !bad && !ring_pass(next, (e - 1) / kSB, wait_stage, leave_stage)) {
      atomicOr(err, 1);
      bad = true;
    }
    bad = __shfl_sync(0xffffffffu, bad, 0);
    if (mine) {
#pragma unroll
      for (int jh = 0; jh < 2; ++jh) {
        l_run[jh] += __shfl_xor_sync(0xffffffffu, l_run[jh], 4);
        l_run[jh] += __shfl_xor_sync(0xffffffffu, l_run[jh], 8);
        l_run[jh] += __shfl_xor_sync(0xffffffffu, l_run[jh], 16);
        if (bad) m_run[jh] = -INFINITY;
      }
    }
    consumer_sync();
    if (mine) {
      float* ws = slot + warp * PW;
#pragma unroll
      for (int i = 0; i < MT; ++i) {
        const int d0 = G * (i / GT) + CPL * gid + 2 * (i % GT);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int h = 2 * tid + (r & 1);
          if (h < grp) ws[h * (D + 2) + 2 + d0 + (r >> 1)] = o[i][r];
        }
      }
      if (gid == 0)
#pragma unroll
        for (int jh = 0; jh < 2; ++jh)
          if (2 * tid + jh < grp) {
            ws[(2 * tid + jh) * (D + 2)] = m_run[jh];
            ws[(2 * tid + jh) * (D + 2) + 1] = l_run[jh];
          }
    }
    consumer_sync();
    const int np = min(kNW, e - a);
    if (tc < grp) {
      float M = -INFINITY;
      for (int i = 0; i < np; ++i) M = fmaxf(M, slot[((a + i) % kNW) * PW + tc * (D + 2)]);
      float L = 0.f;
      for (int i = 0; i < np; ++i) {
        const float* pp = slot + ((a + i) % kNW) * PW + tc * (D + 2);
        const float w = pp[0] == -INFINITY ? 0.f : exp2f(pp[0] - M);
        mg->m[i][tc] = w;
        L += w * pp[1];
      }
      mg->M[tc] = M;
      mg->L[tc] = L;
    }
    consumer_sync();
    const int c0 = cta_of(hs, N, P), c1 = cta_of(hs + nb - 1, N, P);
    const int nct = c1 - c0 + 1;
    if (nct > kFullSlot) {                           // the host sizes the grid so this cannot happen
      if (tc == 0) atomicOr(err, 4);
      continue;
    }
    const int64_t orow0 = (int64_t)b * g.Hq + hkv * grp;
    for (int idx = tc; idx < grp * D; idx += kNW * 32) {
      const int h = idx / D, d = idx % D;
      float acc = 0.f;
      for (int i = 0; i < np; ++i) acc += mg->m[i][h] * slot[((a + i) % kNW) * PW + h * (D + 2) + 2 + d];
      if (nct == 1) qr[h * D + d] = acc;
      else wsb[((orow0 + h) * kMaxSplits + (blockIdx.x - c0)) * (D + kWsStride) + 2 + d] = acc;
    }
    if (nct == 1) {
      finish(b, hkv, mg->M, mg->L);
      continue;
    }
    if (tc < grp) {
      float* wr = wsb + ((orow0 + tc) * kMaxSplits + (blockIdx.x - c0)) * (D + kWsStride);
      wr[0] = mg->M[tc];
      wr[1] = mg->L[tc];
    }
    consumer_sync();
    if (tc == 0) {
      __threadfence();
      mg->last = atomicAdd(&g.counters[hd], 1u) == (unsigned)nct - 1;
    }
    consumer_sync();
    if (!mg->last) continue;
    __threadfence();
    if (tc < grp * nct) {
      const int h = tc / nct, i = tc % nct;
      const float* wr = wsb + ((orow0 + h) * kMaxSplits + i) * (D + kWsStride);
      mg->m[i][h] = __ldcg(wr);
      mg->l[i][h] = __ldcg(wr + 1);
    }
    consumer_sync();
    if (tc < grp) {
      float M = -INFINITY;
      for (int i = 0; i < nct; ++i) M = fmaxf(M, mg->m[i][tc]);
      float L = 0.f;
      for (int i = 0; i < nct; ++i) {
        const float w = mg->m[i][tc] == -INFINITY ? 0.f : exp2f(mg->m[i][tc] - M);
        mg->m[i][tc] = w;
        L += w * mg->l[i][tc];
      }
      mg->M[tc] = M;
      mg->L[tc] = L;
    }
    consumer_sync();
    for (int idx = tc; idx < grp * D; idx += kNW * 32) {
      const int h = idx / D, d = idx % D;
      const float* wr = wsb + (orow0 + h) * kMaxSplits * (D + kWsStride) + 2 + d;
      float acc = 0.f;
#pragma unroll 4
      for (int i = 0; i < nct; ++i) acc += mg->m[i][h] * __ldcg(wr + i * (D + kWsStride));
      qr[h * D + d] = acc;
    }
    if (tc == 0) g.counters[hd] = 0;                 // ready for the next call
    finish(b, hkv, mg->M, mg->L);
  }
}

template <int D, int KB, int VB, int G>
size_t stream_smem(int grp, int* ns) {
  using C = KCfg<D, KB, VB, G>;
  const size_t fixed = (size_t)slot_floats(grp * (D + 2)) * 4 + (size_t)8 * D * 4 + sizeof(Merge);
  int n = (int)((kSmemMax - fixed) / (C::STAGE + 16));
  if (n > kMaxStages) n = kMaxStages;
  *ns = n;
  return (size_t)n * C::STAGE + fixed + (size_t)2 * n * 8;
}

template <int D, int KB, int VB, int G>
cudaError_t launch_t(const Geom& g, const void* q, float scale, int* err, void* out,
                     cudaStream_t s) {
  const int grp = g.Hq / g.H;
  auto full = grp <= 2 ? kvarn_full_kernel<D, 2> : grp <= 4 ? kvarn_full_kernel<D, 4> : kvarn_full_kernel<D, 8>;
  launch_pdl(full, dim3(kFullSplits, g.H, g.B), dim3(kFullWarps * 32), 0, s, g,
             reinterpret_cast<const __nv_bfloat16*>(q), scale);
  int ns = 0;
  const size_t sm = stream_smem<D, KB, VB, G>(grp, &ns);
  auto kern = grp <= 2 ? decode_stream_kvarn_kernel<D, KB, VB, G, true>
                       : decode_stream_kvarn_kernel<D, KB, VB, G, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  launch_pdl(kern, dim3(decode_stream_ctas(g)), dim3(kThreads), sm, s, g,
             reinterpret_cast<const __nv_bfloat16*>(q), scale, (float)(1.0 / sqrt((double)D)), err,
             reinterpret_cast<__nv_bfloat16*>(out), ns);
  return cudaGetLastError();
}

}  // namespace

// Eight heads of 256 leave room for one ring stage only: nothing is copied while a stage
// is worked on, and it still takes a quarter of the split kernel's time (batch 4, 8 kv
// heads, 8300 tokens: 82 us against 357).
bool decode_stream_kvarn_supported(const Geom& g) {
  const bool shape = (g.D == 256 && g.G == 64) || (g.D == 64 && g.G == 32);
  if (!(g.fmt == KVQ_FMT_KVARN && g.act == KVQ_BF16 && shape && g.kb == 4 && g.vb == 2 &&
        g.Hq / g.H <= 8))
    return false;
  int ns = 0;
  if (g.D == 256) stream_smem<256, 4, 2, 64>(g.Hq / g.H, &ns);
  else stream_smem<64, 4, 2, 32>(g.Hq / g.H, &ns);
  return ns >= 1;
}

cudaError_t launch_decode_stream_kvarn(const Geom& g, const void* q, float scale, int* err,
                                       void* out, cudaStream_t s) {
  if (g.D == 256) return launch_t<256, 4, 2, 64>(g, q, scale, err, out, s);
  return launch_t<64, 4, 2, 32>(g, q, scale, err, out, s);
}

}  // namespace kvq
