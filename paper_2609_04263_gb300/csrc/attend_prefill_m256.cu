// Causal GQA prefill attention over the stored reconstruction on the
// 5th-generation tensor cores (tcgen05), Sections 3.1-3.3: the L newest
// queries attend to every token up to their own position, and every key and
// value is the cache's reconstruction (codes x scale + offset, or the
// full-precision residual window of a KIVI cache).
//
// A CTA holds 256 query rows of one (sequence, kv head): the g query heads of the
// kv head x 256/g consecutive queries, head-major, as two 128-row query tiles A
// and B that share every reconstructed key/value tile of 64 tokens.  At head_dim
// 128 two CTAs (a cluster, one MMA pair) share it too: the second's queries follow
// the first's, the MMAs take tile A (or B) of both, and of K each CTA builds 32 of
// the tokens, of V the 64 tokens' half of the channels, which is how a pair shares
// the second operand of its MMAs.  Four roles:
//   loader (warp 13): the packed rows of a tile, a bulk copy per plane;
//   producers (warps 8-11): reconstruct the tile, or the CTA's share of it: K as a
//     bf16 high part (the fp32 value truncated) plus the bf16 of the remainder
//     (about 16 significant bits: large logits need more than bf16's 8), V as fp16
//     computed in packed half2 arithmetic (code x scale + offset, one rounding),
//     into four shared tile buffers in the 128-byte-swizzled K-major layout of the
//     MMA descriptors (V transposed: channels x tokens);
//   issuer (warp 12, of a pair the first CTA's; one lane issues): S_X = Q_X K_hi^T
//     + Q_X K_lo^T into double-buffered TMEM tiles (128 x 64 fp32 in each CTA) and
//     O_X += P_X V into 128 x D fp32 for X = A, B; completions are signalled by
//     tcgen05.commit on mbarriers (of both CTAs);
//   softmax A (warps 0-3) and B (warps 4-7): thread r owns row r of its
//     query tile (TMEM lane r): reads the 64 scores, masks causally, keeps
//     the running maximum m and sum l in log2 units, writes P as fp16 over
//     its S tile.  O is rescaled (in TMEM) only when a row's maximum grows by
//     more than 8 (so P stays <= 2^8 in fp16); the final O / l is stored as
//     bf16.
// The barriers that wake the issuer (tiles built, P written) sit in the first
// CTA and count one arrival per warp.
// What bounds it, per 64-token tile: D = 128, building the tiles, most of 2,700
// cycles (2,300 without building: the MMAs, 1,540, and the waits between them and
// the softmax warps); D = 64, the chain from scores over softmax to P V and the buffers
// it frees, about 2,000 cycles, 1,060 of them softmax.
//   2 x 8192 tokens, 32 / 8 heads of 128, KIVI 2-bit: 2081 us with two tile
// buffers, 1745 with three, 1338 here.  A thread's share of a tile is kept small
// and the issuer holds one copy of each product: with 64 channels of K or V to a
// thread unrolled and five copies the roles' code did not fit the instruction
// cache (1.5 of 10 cycles an instruction went to fetching it), 1,800 us as a pair
// (1,480 with one copy, 1,400 with the build loops rolled up as well).
//   4 x 2029 tokens, 32 / 4 heads of 64, affine 4-bit: 229 us with two tile buffers,
// 199 with four, 179 here.  As a pair 192: less to build, which did not bound it,
// and longer waits.
// Every wait is bounded and also gives up when another role has timed out;
// the issuer drains its MMAs before TMEM is freed, and a timed-out CTA
// stores nothing and sets the library's error word.
#include <math.h>

#include "tc_common.cuh"

namespace kvq {
namespace {
using namespace tc;

constexpr int kM = 128;              // rows per query tile (MMA M)
constexpr int kTok = 64;             // tokens per KV tile
constexpr int kRowsCta = 2 * kM;     // query rows per CTA
constexpr int kProdWarps = 4;
constexpr int kThreads = 14 * 32;    // 8 softmax, 4 producer, 1 issuer, 1 loader warp
constexpr float kRescale = 8.f;      // log2 growth of a row maximum that forces a rescale

// Shared memory (bytes from a 1024-aligned base).
template <int D, int BITS>
struct M256Layout {
  // Two CTAs share each K/V tile where building it bounds the kernel: D = 128 takes
  // 1745 us alone and 1335 paired, D = 64 179 alone and 192 paired (shapes above).
  static constexpr bool PAIR = D == 128;
  static constexpr int KT = PAIR ? kTok / 2 : kTok; // tokens of K per CTA
  static constexpr int VC = PAIR ? D / 2 : D;       // channels of V per CTA
  static constexpr int NP = 32 * kProdWarps;        // producer threads
  static constexpr int KC = KT * D / NP;            // channels of K per thread
  static constexpr int CV = VC * 8 / NP;            // channels of V per thread
  static_assert(KC == 32 && CV == 4, "build_tile: one group of K, one or two code bytes of V a token");
  // score tiles (TMEM) per query tile: what O (2 D columns) leaves of 512
  static constexpr int SB = 2;
  // Reconstructed K/V tile buffers.  A buffer is held from the start of its build to
  // the end of its P V, about three tile times.
  static constexpr int KVB = 4;
  static constexpr int QT = kM * D * 2;             // one query tile: D/64 atoms of 16 KB
  static constexpr int Q_OFF = 0;
  static constexpr int KV_OFF = 2 * QT;
  static constexpr int KH = 0;                      // K hi: D/64 atoms of KT rows x 128 B
  static constexpr int KL = KT * D * 2;             // K lo: the same
  static constexpr int VT = 2 * KT * D * 2;         // V^T: VC rows x 128 B (64 tokens)
  static constexpr int KV_B = VT + VC * 128;
  // packed tile as stored in the cache planes: 64 code rows of K and of V,
  // then four metadata pieces of 4 D bytes each (per-token group scales and
  // offsets of 64 tokens, or KIVI's per-channel scales and offsets of the
  // tile's two 32-token key blocks)
  static constexpr int CROW = D * BITS / 8;         // code bytes per token
  static constexpr int RKC = 0, RVC = kTok * CROW;
  static constexpr int RKS = 2 * kTok * CROW, RKZ = RKS + 4 * D, RVS = RKZ + 4 * D,
                       RVZ = RVS + 4 * D;
  static constexpr int RAW_B = RVZ + 4 * D;
  static constexpr int RAW_OFF = KV_OFF + KVB * KV_B;
  static constexpr int RAW = 3;                     // packed-tile stages (copied ahead)
  static constexpr int KS_OFF = RAW_OFF + RAW * RAW_B;   // KIVI: a key warp's fp32 scales and offsets
  static constexpr int TOTAL = KS_OFF + NP / 32 * 2 * KC * 4;
  static constexpr int ALLOC = TOTAL + 1024;        // alignment slack
  static_assert(ALLOC <= 226 * 1024, "one CTA's shared memory");
};

// The instructions of one CTA or of a pair.
template <bool PAIR>
__device__ __forceinline__ void mma_a_fill(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  if (PAIR) umma_pair_a_fill(d, a, b, id, acc);
  else umma_a_fill(d, a, b, id, acc);
}
template <bool PAIR>
__device__ __forceinline__ void mma_a_lastuse(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  if (PAIR) umma_pair_a_lastuse(d, a, b, id, acc);
  else umma_a_lastuse(d, a, b, id, acc);
}
template <bool PAIR>
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t id, uint32_t acc) {
  if (PAIR) umma_pair_ts(d, a, b, id, acc);
  else umma_ts(d, a, b, id, acc);
}
template <bool PAIR>
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  if (PAIR) umma_commit_pair(bar);
  else umma_commit(bar);
}
template <bool PAIR>
__device__ __forceinline__ void arrive_first(uint64_t* bar) {   // on the first CTA's barrier
  if (PAIR) mbar_arrive_pair(mapa(bar, 0));
  else mbar_arrive(bar);
}
template <bool PAIR>
__device__ __forceinline__ void tmem_alloc512(uint32_t* base) {
  if (PAIR) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  } else {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
}
template <bool PAIR>
__device__ __forceinline__ void tmem_free512(uint32_t tmem) {
  if (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// Bytes of one packed tile the loader copies (codes of K and V, metadata).
template <int D, int BITS, int FMT>
__host__ __device__ constexpr int raw_bytes() {
  return 2 * kTok * (D * BITS / 8) + (FMT == KVQ_FMT_SYMMETRIC ? 2 : 4) * 4 * D;
}

// Loader: the packed rows of tile t0 .. t0 + 63 of every plane the tile
// reads, one bulk copy per plane.  Planes hold whole 64-row tiles (their
// row counts are padded to multiples of 64), so a tile reaching past the
// stored tokens copies rows that are never used.
template <int D, int BITS, int FMT>
__device__ __forceinline__ void load_raw(const Geom& g, int b, int h, int t0, unsigned char* raw,
                                         uint64_t* bar) {
  using S = M256Layout<D, BITS>;
  constexpr uint32_t CB = kTok * S::CROW;
  mbar_expect_tx(bar, raw_bytes<D, BITS, FMT>());
  // a tile is one 64-token page of a paged cache: tok_ptr finds its rows
  bulk_copy(raw + S::RKC, tok_ptr<uint8_t>(g, KVQ_PLANE_K_CODES, b, h, t0), CB, bar);
  bulk_copy(raw + S::RVC, tok_ptr<uint8_t>(g, KVQ_PLANE_V_CODES, b, h, t0), CB, bar);
  // KIVI: two key blocks of D channels
  const __half* ks = FMT == KVQ_FMT_KIVI ? blk_ptr<__half>(g, KVQ_PLANE_K_SCALE, b, h, t0 / 32)
                                         : tok_ptr<__half>(g, KVQ_PLANE_K_SCALE, b, h, t0);
  bulk_copy(raw + S::RKS, ks, 4 * D, bar);
  if (FMT != KVQ_FMT_SYMMETRIC) {
    const __half* kz = FMT == KVQ_FMT_KIVI
                           ? blk_ptr<__half>(g, KVQ_PLANE_K_ZERO, b, h, t0 / 32)
                           : tok_ptr<__half>(g, KVQ_PLANE_K_ZERO, b, h, t0);
    bulk_copy(raw + S::RKZ, kz, 4 * D, bar);
  }
  bulk_copy(raw + S::RVS, tok_ptr<__half>(g, KVQ_PLANE_V_SCALE, b, h, t0), 4 * D, bar);
  if (FMT != KVQ_FMT_SYMMETRIC)
    bulk_copy(raw + S::RVZ, tok_ptr<__half>(g, KVQ_PLANE_V_ZERO, b, h, t0), 4 * D, bar);
}

// K: 8 channels reconstructed in fp32 and split into a bf16 high part (the
// value truncated) and the bf16 of the remainder.
__device__ __forceinline__ void split_store(const uint64_t (&k2)[4], unsigned char* hi_dst,
                                            unsigned char* lo_dst) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float a, c;
    f2unpack(k2[i], a, c);
    const uint32_t ab = __float_as_uint(a) & 0xFFFF0000u, cb = __float_as_uint(c) & 0xFFFF0000u;
    h[i] = __byte_perm(ab, cb, 0x7632);
    float ra, rc;
    f2unpack(fadd2(k2[i], f2pack(-__uint_as_float(ab), -__uint_as_float(cb))), ra, rc);
    l[i] = pack_bf16(ra, rc);
  }
  *reinterpret_cast<uint4*>(hi_dst) = make_uint4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<uint4*>(lo_dst) = make_uint4(l[0], l[1], l[2], l[3]);
}

// Producers: reconstruct this CTA's share of the K and V operand tiles of KV tile
// t0 from the packed tile in `raw` (tokens below tq), the KIVI residual ring
// (tq <= t < T) or zeros (t >= T).  tid 0..127:
//   K: thread (tk = tid % KT, hf = tid / KT): token KT rank + tk, channels
//      KC hf .. KC hf + KC - 1.
//   V: thread (tb = tid % 8, vq = tid % NP / 8): tokens 8 tb .. 8 tb + 7 and
//      channels CV vq .. CV vq + CV - 1 of this CTA's, in half2 arithmetic, stored
//      as rows of the transposed tile (half a 16-byte chunk per row and trip).
template <int D, int BITS, int FMT>
__device__ __forceinline__ void build_tile(const Geom& g, int b, int h, int t0, int T, int tq,
                                           int tid, int rank, const unsigned char* raw, float* ksz,
                                           unsigned char* kv) {
  using S = M256Layout<D, BITS>;
  constexpr bool KIVI = FMT == KVQ_FMT_KIVI;
  constexpr bool SYM = FMT == KVQ_FMT_SYMMETRIC;
  constexpr int CV = S::CV;
  constexpr int NCH = S::KC / 8;                  // K chunks of 8 channels per thread
  constexpr int NKW = S::KC * BITS / 32;          // K code words per thread
  {
  // ---- K tile ----
  const int tk = tid % S::KT, hf = tid / S::KT, tt = rank * S::KT + tk;
  const int t = t0 + tt;
  // KIVI: the warp's tokens are one block; its scales and offsets of the warp's
  // channels are converted once (a lane one or two channels) and read back as fp32.
  // Converted by every lane for its own token, 128 conversions a tile kept the unit
  // that also serves the softmax warps' exponentials busy (2,282 us against
  // 1,796, shape above, in the version with 64 channels to a thread).
  float* kf = ksz + (tid >> 5) * (2 * S::KC);
  if constexpr (KIVI) {
    __syncwarp();                                  // the previous tile's are read
#pragma unroll
    for (int i = 0; i < S::KC / 32; ++i) {
      const int e = 32 * i + (tid & 31);
      const __half* sp = reinterpret_cast<const __half*>(raw + S::RKS) + (tt >> 5) * D + hf * S::KC + e;
      kf[e] = __half2float(sp[0]);
      kf[S::KC + e] = __half2float(sp[(S::RKZ - S::RKS) / 2]);
    }
    __syncwarp();
  }
  if (t < tq) {
    uint32_t kw[NKW];
    const unsigned char* cp = raw + S::RKC + tt * S::CROW + hf * (S::KC * BITS / 8);
    if constexpr (NKW >= 4) {
#pragma unroll
      for (int i = 0; i < NKW / 4; ++i) {
        const uint4 u = *reinterpret_cast<const uint4*>(cp + 16 * i);
        kw[4 * i] = u.x; kw[4 * i + 1] = u.y; kw[4 * i + 2] = u.z; kw[4 * i + 3] = u.w;
      }
    } else {
      const uint2 u = *reinterpret_cast<const uint2*>(cp);
      kw[0] = u.x; kw[1] = u.y;
    }
    uint32_t ks = 0, kz = 0;                      // affine/symmetric: the group's metadata
    if constexpr (!KIVI) {
      const unsigned char* sp = raw + S::RKS + tt * (D / 16) + hf * (S::KC / 16);
      ks = *reinterpret_cast<const unsigned short*>(sp);
      if (!SYM) kz = *reinterpret_cast<const unsigned short*>(sp + (S::RKZ - S::RKS));
    }
    const uint64_t bias2 = f2pack(-8388608.f, -8388608.f);
    constexpr int WT = BITS / 2;                  // code words per trip
#pragma unroll
    for (int c0 = 0; c0 < NCH; c0 += 2) {
      uint32_t cw[WT];
#pragma unroll
      for (int i = 0; i < WT; ++i) cw[i] = kw[i];
#pragma unroll
      for (int i = 0; i + WT < NKW; ++i) kw[i] = kw[i + WT];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int c = c0 + u, cc = hf * NCH + c;    // chunk along D
      const uint32_t w = BITS == 4 ? cw[u * (WT - 1)] : cw[0] >> (16 * u);
      uint64_t k2[4];
      if constexpr (KIVI) {
        const float4* sp = reinterpret_cast<const float4*>(kf + 8 * c);
        const float4* zp = reinterpret_cast<const float4*>(kf + S::KC + 8 * c);
        const float4 sv[2] = {sp[0], sp[1]}, zv[2] = {zp[0], zp[1]};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 sq = sv[i / 2], zq = zv[i / 2];
          const uint64_t c2 = fadd2(f2pack(code_biased<BITS>(w, 2 * i), code_biased<BITS>(w, 2 * i + 1)), bias2);
          k2[i] = i & 1 ? ffma2(c2, f2pack(sq.z, sq.w), f2pack(zq.z, zq.w))
                        : ffma2(c2, f2pack(sq.x, sq.y), f2pack(zq.x, zq.y));
        }
      } else {
        const float s = __half2float(__ushort_as_half((unsigned short)ks));
        const float m = SYM ? -(float)(1 << (BITS - 1)) * s : __half2float(__ushort_as_half((unsigned short)kz));
        const uint64_t ss = f2pack(s, s), mm = f2pack(m, m);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint64_t c2 = fadd2(f2pack(code_biased<BITS>(w, 2 * i), code_biased<BITS>(w, 2 * i + 1)), bias2);
          k2[i] = ffma2(c2, ss, mm);
        }
      }
      unsigned char* base = kv + (cc >> 3) * (S::KT * 128);
      split_store(k2, base + S::KH + sw128(tk, cc & 7), base + S::KL + sw128(tk, cc & 7));
    }
    }
  } else {
    // KIVI residual window (full precision) or beyond the cache (zeros)
#pragma unroll 1
    for (int c = 0; c < NCH; ++c) {
      const int cc = hf * NCH + c;
      uint4 u = make_uint4(0, 0, 0, 0);
      if (KIVI && t < T)
        u = *reinterpret_cast<const uint4*>(
            plane_ptr<__nv_bfloat16>(g, KVQ_PLANE_K_FULL, b, h, t % g.ring, 8 * cc));
      unsigned char* base = kv + (cc >> 3) * (S::KT * 128);
      *reinterpret_cast<uint4*>(base + S::KH + sw128(tk, cc & 7)) = u;
      *reinterpret_cast<uint4*>(base + S::KL + sw128(tk, cc & 7)) = make_uint4(0, 0, 0, 0);
    }
  }
  }
  // ---- V^T tile: rows CV vq + e, 16-byte chunk tb (tokens 8 tb ..) ----
  const int tb = tid & 7, vq = tid % S::NP >> 3;
  const int ch = rank * S::VC + vq * CV, grp_v = ch / 32;
  const __half2 bias = __float2half2_rn(1024.f);
#pragma unroll
  for (int p0 = 0; p0 < 4; p0 += 2) {             // tokens 2 p0 .. 2 p0 + 3
  uint32_t out[CV][2];
#pragma unroll
  for (int pp = 0; pp < 2; ++pp) {                // token pair (2p, 2p + 1)
    const int p = p0 + pp;
    uint32_t w2[2], s2u, z2u;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int tv = 8 * tb + 2 * p + u;          // token within the tile
      const unsigned char* cp = raw + S::RVC + tv * S::CROW + ch * BITS / 8;
      if constexpr (BITS == 4) w2[u] = *reinterpret_cast<const unsigned short*>(cp);
      else w2[u] = *cp;
    }
    {
      const int tv = 8 * tb + 2 * p;
      const unsigned short* sp = reinterpret_cast<const unsigned short*>(raw + S::RVS) + tv * (D / 32) + grp_v;
      s2u = (uint32_t)sp[0] | ((uint32_t)sp[D / 32] << 16);
      if constexpr (SYM) {
        const __half2 z = __hmul2(*reinterpret_cast<const __half2*>(&s2u),
                                  __float2half2_rn(-(float)(1 << (BITS - 1))));
        z2u = *reinterpret_cast<const uint32_t*>(&z);
      } else {
        const unsigned short* zp = reinterpret_cast<const unsigned short*>(raw + S::RVZ) + tv * (D / 32) + grp_v;
        z2u = (uint32_t)zp[0] | ((uint32_t)zp[D / 32] << 16);
      }
    }
    const uint32_t pw = w2[0] | (w2[1] << 16);
    const __half2 s2 = *reinterpret_cast<const __half2*>(&s2u);
    const __half2 z2 = *reinterpret_cast<const __half2*>(&z2u);
#pragma unroll
    for (int e = 0; e < CV; ++e) {
      constexpr uint32_t m2 = ((1u << BITS) - 1) * 0x00010001u;
      const uint32_t x = ((pw >> (e * BITS)) & m2) | 0x64006400u;
      const __half2 c2 = __hsub2(*reinterpret_cast<const __half2*>(&x), bias);
      const __half2 v2 = __hfma2(s2, c2, z2);
      out[e][pp] = *reinterpret_cast<const uint32_t*>(&v2);
    }
  }
  // tokens of the KIVI residual window, or beyond the cache, replace theirs
  const int tv0 = t0 + 8 * tb + 2 * p0;
  if (tv0 + 3 >= tq) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int tv = tv0 + i;
      if (tv < tq) continue;
      __nv_bfloat16 vals[CV];
      if (KIVI && tv < T) {
        const __nv_bfloat16* src = plane_ptr<__nv_bfloat16>(g, KVQ_PLANE_V_FULL, b, h, tv % g.ring, ch);
        const uint2 u = *reinterpret_cast<const uint2*>(src);
        memcpy(vals, &u, sizeof(vals));
      } else {
#pragma unroll
        for (int e = 0; e < CV; ++e) vals[e] = __float2bfloat16_rn(0.f);
      }
#pragma unroll
      for (int e = 0; e < CV; ++e) {
        const uint32_t hv = __half_as_ushort(__float2half_rn(__bfloat162float(vals[e])));
        out[e][i >> 1] = (i & 1) ? ((out[e][i >> 1] & 0xFFFFu) | (hv << 16))
                                 : ((out[e][i >> 1] & 0xFFFF0000u) | hv);
      }
    }
  }
#pragma unroll
  for (int e = 0; e < CV; ++e)
    *reinterpret_cast<uint2*>(kv + S::VT + sw128(CV * vq + e, tb) + 4 * p0) = make_uint2(out[e][0], out[e][1]);
  }
}

template <int D, int BITS, int FMT>
__global__ void __launch_bounds__(kThreads, 1)
attend_prefill_m256_kernel(Geom g, const __nv_bfloat16* __restrict__ q, int L, float scale,
                           __nv_bfloat16* __restrict__ out, int nq, int* err) {
  pdl_wait();
  pdl_trigger();
  using S = M256Layout<D, BITS>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t raw_full[S::RAW], raw_free[S::RAW], kv_full[S::KVB], kv_free[S::KVB],
      s_full[2][S::SB], p_full[2][S::SB], s_free[2][S::SB], done_bar;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int NC = S::PAIR ? 2 : 1;                  // CTAs that share a K/V tile
  const uint32_t rank = S::PAIR ? cluster_rank() : 0;
  const int qset = (gridDim.x - 1 - blockIdx.x) / NC;  // longest first
  const int hkv = blockIdx.y, b = blockIdx.z;
  const int grp = g.Hq / g.H;
  const int T = seq_tokens(g, b);
  const int tq = FMT == KVQ_FMT_KIVI ? kivi_tq(T, g.R, g.G) : T;
  // a ragged cache's sequence b attends the rows of its last append
  const int Lb = g.layout == KVQ_LAYOUT_UNIFORM ? L : g.seq_new[b];
  if (NC * qset * nq >= Lb) return;                    // no query of this sequence here
  const int q0 = (NC * qset + (int)rank) * nq;
  const int nql = min(nq, Lb - q0);                    // <= 0: no query here, only a share of K/V
  const int pos_first = T - Lb + q0;
  const int t_end = T - Lb + min(NC * (qset + 1) * nq, Lb);   // keys [0, t_end), the pair's
  const int ntiles = (t_end + kTok - 1) / kTok;
  volatile int* abort = &abort_flag;

  if (threadIdx.x == 0) {
    for (int i = 0; i < S::RAW; ++i) {
      mbar_init(&raw_full[i], 1);
      mbar_init(&raw_free[i], kProdWarps);
    }
    for (int i = 0; i < S::KVB; ++i) {
      mbar_init(&kv_full[i], NC * kProdWarps);
      mbar_init(&kv_free[i], 1);
    }
    for (int x = 0; x < 2; ++x)
      for (int i = 0; i < S::SB; ++i) {
        mbar_init(&s_full[x][i], 1);
        mbar_init(&p_full[x][i], NC * (kM / 32));
        mbar_init(&s_free[x][i], 1);
      }
    mbar_init(&done_bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 12) {
    tmem_alloc512<S::PAIR>(&tmem_base);
  }
  // queries -> the swizzled Q tiles (softmax threads, one row each)
  const int row = threadIdx.x;                          // 0..255 for the softmax roles
  int pos = -1;
  if (warp < 8) {
    const int hl = row / nq, qi = row % nq;
    const bool valid = hl < grp && qi < nql;
    if (valid) pos = pos_first + qi;
    const __nv_bfloat16* src = q + (((int64_t)b * g.Hq + hkv * grp + hl) * L + q0 + qi) * D;
    unsigned char* qt = smem + S::Q_OFF + (row >> 7) * S::QT;
    const int r = row & 127;
#pragma unroll
    for (int c = 0; c < D / 8; ++c) {
      uint4 v = make_uint4(0, 0, 0, 0);
      if (valid) v = *reinterpret_cast<const uint4*>(src + 8 * c);
      *reinterpret_cast<uint4*>(qt + (c >> 3) * (kM * 128) + sw128(r, c & 7)) = v;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  if (S::PAIR) cluster_sync();                         // both CTAs' barriers are set up
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;

  if (warp == 13) {
    // ---------------- loader: packed tiles into the raw ring ----------------
    if (lane == 0) {
      int issued = 0;
      for (int j = 0; j < ntiles; ++j) {
        const int st = j % S::RAW;
        if (j >= S::RAW && !mbar_wait_or_abort(&raw_free[st], ((j - S::RAW) / S::RAW) & 1, abort)) break;
        load_raw<D, BITS, FMT>(g, b, hkv, j * kTok, smem + S::RAW_OFF + st * S::RAW_B,
                               &raw_full[st]);
        issued = j + 1;
      }
      // no copy may still be landing in shared memory when the CTA exits
      // (after a timeout the producers stop consuming): wait, bounded, for
      // the last tile issued on each stage
      for (int t = issued > S::RAW ? issued - S::RAW : 0; t < issued; ++t)
        if (!mbar_wait(&raw_full[t % S::RAW], (t / S::RAW) & 1)) *abort = 1;
    }
  } else if (warp >= 8 && warp < 12) {
    // ---------------- producers: reconstruct K and V tiles ----------------
    const int tid = threadIdx.x - 256;
    for (int j = 0; j < ntiles; ++j) {
      const int st = j % S::RAW, kb = j % S::KVB;
      bool ok = mbar_wait_or_abort(&raw_full[st], (j / S::RAW) & 1, abort);
      ok = ok && (j < S::KVB ||
                  mbar_wait_or_abort(&kv_free[kb], ((j - S::KVB) / S::KVB) & 1, abort));
      if (!__all_sync(0xffffffffu, ok)) break;
      unsigned char* kv = smem + S::KV_OFF + kb * S::KV_B;
      build_tile<D, BITS, FMT>(g, b, hkv, j * kTok, T, tq, tid, (int)rank,
                               smem + S::RAW_OFF + st * S::RAW_B,
                               reinterpret_cast<float*>(smem + S::KS_OFF), kv);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // for the MMAs' reads
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&raw_free[st]);
        arrive_first<S::PAIR>(&kv_full[kb]);
      }
    }
  } else if (warp == 12) {
    if (rank == 0) {
      // ---------------- MMA issuer ----------------
      // For each query tile X in turn Q_X K^T of a later tile, then P_X V of tile
      // j, each blocking on the barrier it needs: what Q_X K^T waits for, P_X V of
      // an earlier tile, is two steps of the other query tile back, so the tensor
      // pipe has work meanwhile.  While that later tile is not built yet, P V
      // goes first (D = 128).  An issuer that polled for whichever came first answered
      // several hundred cycles late, twice in the chain of every tile (D = 64: 199 us,
      // 179 so).  The whole warp runs the loop (its values stay
      // warp-uniform) and one elected lane issues the MMAs and their commits.
      // Descriptors are formed once: a K step of 16 elements advances the start
      // address by 32 bytes (2 in the descriptor's 16-byte units).
      constexpr uint32_t id_qk = idesc_bf16(NC * kM, kTok);
      constexpr uint32_t id_pv = idesc_f16(NC * kM, D);
      const uint64_t qdesc0 = sw128_desc(smem + S::Q_OFF);
      const uint64_t kvdesc0 = sw128_desc(smem + S::KV_OFF);   // K/V buffer b: + b KV_B / 16
      const bool leader = elect_one();
      auto qk = [&](int x, int j) -> bool {
        const int kb = j % S::KVB, bf = j % S::SB;
        if ((x == 0 && !warp_wait(&kv_full[kb], (j / S::KVB) & 1, abort)) ||
            (j >= S::SB && !warp_wait(&s_free[x][bf], ((j - S::SB) / S::SB) & 1, abort)))
          return false;
        tc_fence_after();
        if (leader) {
          const uint32_t ts = tmem + (x * S::SB + bf) * kTok;
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            // Q atom: 128 rows x 128 B (1024 units); K atom: KT rows x 128 B (8 KT units)
            const uint64_t qd = qdesc0 + (uint64_t)(x * (S::QT >> 4) + (kk >> 2) * 1024 + (kk & 3) * 2);
            const uint64_t kd = kvdesc0 + (uint64_t)(kb * (S::KV_B >> 4) + (kk >> 2) * (8 * S::KT) + (kk & 3) * 2);
            mma_a_fill<S::PAIR>(ts, qd, kd + (S::KH >> 4), id_qk, kk > 0);   // Q read once
            mma_a_lastuse<S::PAIR>(ts, qd, kd + (S::KL >> 4), id_qk, 1);     // for K hi and lo
          }
          mma_commit<S::PAIR>(&s_full[x][bf]);
        }
        __syncwarp();
        return true;
      };
      auto pv = [&](int x, int j) -> bool {
        const int kb = j % S::KVB, bf = j % S::SB;
        if (!warp_wait(&p_full[x][bf], (j / S::SB) & 1, abort)) return false;
        tc_fence_after();
        if (leader) {
          const uint32_t tp = tmem + (x * S::SB + bf) * kTok;   // P (fp16 pairs) over S's columns
          const uint32_t to = tmem + 2 * S::SB * kTok + x * D;
#pragma unroll
          for (int kk = 0; kk < kTok / 16; ++kk)
            mma_ts<S::PAIR>(to, tp + kk * 8, kvdesc0 + (uint64_t)(kb * (S::KV_B >> 4) + (S::VT >> 4) + kk * 2),
                         id_pv, (j > 0 || kk > 0) ? 1u : 0u);
          mma_commit<S::PAIR>(&s_free[x][bf]);           // S/P buffer free, and O holds tile j
          if (x == 1) mma_commit<S::PAIR>(&kv_free[kb]); // both query tiles done with it
        }
        __syncwarp();
        return true;
      };
      bool ok = true;
#pragma unroll 1
      for (int j = -1; j < ntiles && ok; ++j) {
        const int n = j + 1;
        if constexpr (!S::PAIR) {
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            if (ok && n < ntiles) ok = qk(x, n);
            if (ok && j >= 0) ok = pv(x, j);
          }
        } else {
          bool first = n < ntiles;             // Q K^T of tile n before P V of tile j
          if (first && j >= 0) {
            if (lane == 0) first = mbar_test(&kv_full[n % S::KVB], (n / S::KVB) & 1);
            first = __shfl_sync(0xffffffffu, first, 0);
          }
          // four steps: Q K^T and P V of A, then of B; or both P V, then both Q K^T
#pragma unroll 1                               // one copy of each in the instruction cache
          for (int i = 0; i < 4 && ok; ++i) {
            const bool is_qk = first ? (i & 1) == 0 : i >= 2;
            const int x = first ? i >> 1 : i & 1;
            if (is_qk) ok = n >= ntiles || qk(x, n);
            else ok = j < 0 || pv(x, j);
          }
        }
      }
      if (leader) mma_commit<S::PAIR>(&done_bar);   // every MMA issued above has completed
      if (lane == 0 && !mbar_wait(&done_bar, 0)) *abort = 1;
      __syncwarp();
    }
  } else if (warp < 8) {
    // ---------------- softmax: one row per thread ----------------
    const int x = warp >> 2;                   // query tile
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t s_col = tmem + lane_base + x * S::SB * kTok;
    const uint32_t o_col = tmem + lane_base + 2 * S::SB * kTok + x * D;
    const float c2 = scale * 1.4426950408889634f;   // scores in log2 units
    const uint64_t c22 = f2pack(c2, c2);
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int j = 0; j < ntiles; ++j) {
      const int bf = j % S::SB, t0 = j * kTok;
      // The second CTA of a pair first for the P V that freed this buffer, so that the waits
      // on s_free below skip none of its phases (a parity tells a phase only from its
      // neighbours).  The first CTA's issuer saw that phase end before it issued these
      // scores; that the second hears of it before it hears of them is not given.
      if ((rank == 1 && j >= S::SB && !warp_wait(&s_free[x][bf], ((j - S::SB) / S::SB) & 1, abort)) ||
          !warp_wait(&s_full[x][bf], (j / S::SB) & 1, abort)) {
        ok = false;
        break;
      }
      tc_fence_after();
      uint32_t sr[kTok];
#pragma unroll
      for (int c = 0; c < kTok; c += 16) tmem_ld16_nowait(s_col + bf * kTok + c, sr + c);
      tmem_wait_ld();
      const bool full = t0 + kTok - 1 <= pos;  // no key of the tile is masked
      if (!full) {
#pragma unroll
        for (int i = 0; i < kTok; ++i)
          if (t0 + i > pos) sr[i] = __float_as_uint(-INFINITY);
      }
      // row maximum: four independent chains of three-input maxima over
      // 16 scores each
      float mx4[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const uint32_t* v = sr + 16 * a;
        float mv = fmax3(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]));
#pragma unroll
        for (int k = 3; k < 15; k += 2)
          mv = fmax3(mv, __uint_as_float(v[k]), __uint_as_float(v[k + 1]));
        mx4[a] = fmaxf(mv, __uint_as_float(v[15]));
      }
      const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      const float m_new = fmaxf(m, mx * c2);   // (c2 > 0: the maximum commutes)
      if (j == 0) {
        m = m_new;
      } else if (__any_sync(0xffffffffu, m_new > m + kRescale)) {
        // O is rewritten: the P V of tile j - 1 must have completed
        if (!warp_wait(&s_free[x][(j - 1) % S::SB], ((j - 1) / S::SB) & 1, abort)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const float alpha = m_new > m ? ex2_approx(m - m_new) : 1.f;
        if (m_new > m) {
          l *= alpha;
          m = m_new;
        }
#pragma unroll 1
        for (int c = 0; c < D; c += 16) {
          uint32_t o[16];
          tmem_ld16_nowait(o_col + c, o);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
          tmem_st16(o_col + c, o);
        }
      }
      // P = 2^(s c2 - m) as fp16 pairs over the first 32 columns of this S
      // buffer (masked keys hold -inf: 2^-inf = 0; a row without any visible
      // key so far has m = -inf and keeps P = 0)
      const bool live = m != -INFINITY;
      const uint64_t negm = f2pack(-m, -m);
      uint64_t sum2 = f2pack(0.f, 0.f);
      uint32_t pk[kTok / 2];
#pragma unroll
      for (int i = 0; i < kTok; i += 2) {
        float a0, a1;
        f2unpack(ffma2(f2pack(__uint_as_float(sr[i]), __uint_as_float(sr[i + 1])), c22, negm), a0, a1);
        float p0 = ex2_approx(a0), p1 = ex2_approx(a1);
        if (!live) p0 = p1 = 0.f;
        sum2 = fadd2(sum2, f2pack(p0, p1));
        pk[i / 2] = pack_h2(p0, p1);
      }
      tmem_st16(s_col + bf * kTok, pk);
      tmem_st16(s_col + bf * kTok + 16, pk + 16);
      float s0, s1;
      f2unpack(sum2, s0, s1);
      l += s0 + s1;
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_first<S::PAIR>(&p_full[x][bf]);
    }
    // ---------------- epilogue ----------------
    if (ok && ntiles > 0 &&
        !warp_wait(&s_free[x][(ntiles - 1) % S::SB], ((ntiles - 1) / S::SB) & 1, abort))
      ok = false;
    if (__all_sync(0xffffffffu, ok && !*abort)) {
      tc_fence_after();
      const float inv = l > 0.f ? 1.f / l : 0.f;
      const int hl = row / nq, qi = row % nq;
      __nv_bfloat16* dst = out + (((int64_t)b * g.Hq + hkv * grp + hl) * L + q0 + qi) * D;
#pragma unroll 1
      for (int c = 0; c < D; c += 16) {
        uint32_t o[16];
        tmem_ld16_nowait(o_col + c, o);
        tmem_wait_ld();
        if (pos >= 0) {
          uint32_t w[8];
#pragma unroll
          for (int i = 0; i < 8; ++i)
            w[i] = pack_bf16(__uint_as_float(o[2 * i]) * inv, __uint_as_float(o[2 * i + 1]) * inv);
          *reinterpret_cast<uint4*>(dst + c) = make_uint4(w[0], w[1], w[2], w[3]);
          *reinterpret_cast<uint4*>(dst + c + 8) = make_uint4(w[4], w[5], w[6], w[7]);
        }
      }
    }
  }
  // the issuer's last arrival on the second CTA's barriers has landed
  if (warp == 12 && lane == 0 && rank == 1 && !mbar_wait(&done_bar, 0)) *abort = 1;
  tc_fence_before();
  if (S::PAIR) cluster_sync();                         // neither CTA's TMEM or shared memory is in use
  else __syncthreads();
  if (threadIdx.x == 0 && *abort) atomicOr(err, 8);
  if (warp == 12) {
    tc_fence_after();
    tmem_free512<S::PAIR>(tmem);
  }
}

template <int D, int BITS, int FMT>
cudaError_t launch_m256(const Geom& g, const void* q, int L, float scale, void* out, int* err,
                        cudaStream_t s) {
  auto kern = attend_prefill_m256_kernel<D, BITS, FMT>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       M256Layout<D, BITS>::ALLOC);
  if (e != cudaSuccess) return e;
  const int nq = kRowsCta / (g.Hq / g.H);
  constexpr int NC = M256Layout<D, BITS>::PAIR ? 2 : 1;
  const dim3 grid((L + NC * nq - 1) / (NC * nq) * NC, g.H, g.B);
  const auto start = [&](auto launcher) {
    return launcher(kern, grid, dim3(kThreads), (size_t)M256Layout<D, BITS>::ALLOC, s, g,
                    reinterpret_cast<const __nv_bfloat16*>(q), L, scale,
                    reinterpret_cast<__nv_bfloat16*>(out), nq, err);
  };
  if (NC == 2) start([](auto... a) { return launch_pdl_pair(a...); });
  else start([](auto... a) { return launch_pdl(a...); });
  return cudaGetLastError();
}

template <int D>
cudaError_t launch_m256_d(const Geom& g, const void* q, int L, float scale, void* out, int* err,
                          cudaStream_t s) {
  if (g.fmt == KVQ_FMT_KIVI)
    return g.kb == 4 ? launch_m256<D, 4, KVQ_FMT_KIVI>(g, q, L, scale, out, err, s)
                     : launch_m256<D, 2, KVQ_FMT_KIVI>(g, q, L, scale, out, err, s);
  if (g.fmt == KVQ_FMT_SYMMETRIC)
    return g.kb == 4 ? launch_m256<D, 4, KVQ_FMT_SYMMETRIC>(g, q, L, scale, out, err, s)
                     : launch_m256<D, 2, KVQ_FMT_SYMMETRIC>(g, q, L, scale, out, err, s);
  return g.kb == 4 ? launch_m256<D, 4, KVQ_FMT_AFFINE>(g, q, L, scale, out, err, s)
                   : launch_m256<D, 2, KVQ_FMT_AFFINE>(g, q, L, scale, out, err, s);
}

}  // namespace

// bf16 affine/symmetric/KIVI caches with equal 2- or 4-bit key and value
// codes, G = 32 (KIVI: 32-token key blocks), head_dim 64 or 128, GQA group <= 256.
bool prefill_m256_supported(const Geom& g) {
  const bool fmt_ok = g.fmt == KVQ_FMT_AFFINE || g.fmt == KVQ_FMT_SYMMETRIC || g.fmt == KVQ_FMT_KIVI;
  return fmt_ok && g.act == KVQ_BF16 && (g.D == 64 || g.D == 128) && g.G == 32 && g.kb == g.vb &&
         (g.kb == 2 || g.kb == 4) && g.Hq / g.H <= kRowsCta;
}

cudaError_t launch_prefill_m256(const Geom& g, const void* q, int L, float scale, void* out,
                                int* err, cudaStream_t s) {
  if (g.D == 64) return launch_m256_d<64>(g, q, L, scale, out, err, s);
  return launch_m256_d<128>(g, q, L, scale, out, err, s);
}

}  // namespace kvq
