// Causal GQA prefill attention over a KVarN cache at head_dim 256 on the
// 5th-generation tensor cores (tcgen05), Sections 3.1-3.3, in the
// Hadamard-rotated basis: coded tokens are stored rotated (r_t c_j (s code + m)
// with row scale r_t and per-block column scale c_j), the queries are rotated
// once and the output is rotated back; sinks and staged tokens (stored in the
// original basis) are rotated forward as their tiles are built.
//
// Two CTAs (a cluster, one MMA pair) hold 128 query rows each of one (sequence,
// kv head): the g query heads of the kv head x 128/g consecutive queries, the
// second CTA's following the first's.  Keys and values stream in tiles of 64
// tokens that the two build together: of K each CTA 32 of the tokens, of V the
// 64 tokens' half of the channels, which is how a pair of CTAs shares the second
// operand of its MMAs.  Three roles:
//   producers: reconstruct their share in fp32 into three shared buffers, K
//     (warps 4-7) as a bf16 high part (the value rounded: a truncated one would leave
//     a remainder of one bit more) plus the bf16 of the remainder, V (warps 8-11) rounded to fp16 and transposed (channels x
//     tokens).  A key warp builds 64 channels, a lane one token; a value warp 32
//     channels, a lane two neighbouring tokens (one 32-bit store each channel).
//     The packed words and scales of the next tile are loaded into registers
//     before the current one is built, the tile's column scales go through a
//     small shared array per warp;
//   issuer (warp 12 of the first CTA, one lane issues): S = Q_hi K_hi^T +
//     Q_hi K_lo^T + Q_lo K_hi^T (a rotated query needs more than bf16's 8 bits
//     too) into two TMEM tiles of 128 x 64 fp32 in each CTA, and O += P V into
//     128 x 256 fp32; S runs up to two tiles ahead of P V;
//   softmax (warps 0-3): thread r owns row r (TMEM lane r): 64 scores, causal
//     mask, running maximum and sum in log2 units, P as fp16 over its S tile; O
//     is rescaled only when a row's maximum grows by more than 8.
// The barriers that wake the issuer (tiles built, P written) sit in the first
// CTA and count one arrival per warp of both; the issuer's commits arrive on both
// CTAs' barriers.
//
// Space decides the layout: at D = 256 a 128-row query tile is 64 KB and has two
// parts.  Q_hi stays in shared memory (the MMAs read it once per K step for
// both K parts), Q_lo in 128 TMEM columns next to O's 256 and S's 2 x 64; that
// leaves shared memory for three 48 KB shares of K/V tiles.
// What bounds it: a 64-token tile takes about 2,800 cycles, the MMAs 2,050 of them;
// with two score buffers Q K^T of a tile starts when P V of the tile two before it
// has completed, so the pipe idles while that is signalled, and building the tiles
// (1,850 cycles of each producer warp) slows the chain (2,700 cycles without it).
// A CTA's start and end (rotating queries, sinks and output rows) take 50,000
// cycles.  8192 tokens, 16 query heads, 8 kv heads, one sequence: 7667 us on
// mma.sync (64 rows a CTA, 16-token tiles reconstructed by all its warps), 1526
// with one CTA building 32-token tiles of K and V for 128 rows, 827 here: 1,480 as
// a pair, 1,380 with arrivals that do not wait (mbar_arrive_pair), 1,100 with the
// packed tile loaded without a branch that divides the warp (load_packed) and
// rows of sinks, queries and outputs loaded together, 994 with K and V built by
// warps of their own (no spills), 898 with four rows to a warp in the rotation,
// 818 with the issuer blocking instead of polling, 827 with the second CTA's softmax
// waiting for every phase.
// Every wait is bounded and also gives up when another role has timed out;
// the issuer drains its MMAs before TMEM is freed, and a timed-out CTA stores
// nothing and sets the library's error word.
#include <math.h>

#include "tc_common.cuh"

namespace kvq {
namespace {
using namespace tc;

constexpr int kD = 256;
constexpr int kM = 128;              // query rows per CTA (half of the pair's MMA M)
constexpr int kTok = 64;             // tokens per KV tile
constexpr int kHalf = 32;            // tokens of K per CTA
constexpr int kG = 64;               // block length and group size
constexpr int kProdWarps = 8;
constexpr int kThreads = (4 + kProdWarps + 1) * 32;
constexpr int kKvBufs = 3;
constexpr int kSBufs = 2;
constexpr float kRescale = 8.f;      // log2 growth of a row maximum that forces a rescale

// Shared memory (bytes from a 1024-aligned base).
constexpr int kQOff = 0;                               // Q_hi: 4 atoms of 128 rows x 128 B
constexpr int kKvOff = kM * kD * 2;
constexpr int kKH = 0;                                 // K hi: 4 atoms of 32 rows x 128 B
constexpr int kKL = kHalf * kD * 2;                    // K lo: the same
constexpr int kVT = 2 * kHalf * kD * 2;                // V^T: 128 channels x 128 B
constexpr int kKvB = kVT + kD / 2 * kTok * 2;
constexpr int kColOff = kKvOff + kKvBufs * kKvB;       // per producer warp: 64 column scales
constexpr int kTotal = kColOff + kProdWarps * 64 * 4;
constexpr int kAlloc = kTotal + 1024;                  // alignment slack
constexpr int kQlPitch = kD * 2 + 16;                  // Q_lo rows staged in the K/V area
static_assert(kM * kQlPitch <= kKvBufs * kKvB, "Q_lo rows fit the K/V area");
constexpr int kOPitch = kD + 4;                        // fp32 output rows over Q and K/V
static_assert(kM * kOPitch * 4 <= kTotal, "output rows fit");
static_assert(kAlloc <= 227 * 1024, "one CTA's shared memory");

// TMEM columns: O, Q_lo (two bf16 per column), S tiles (P over them).
constexpr int kTmO = 0, kTmQ = 256, kTmS = 384;

// Four rows of 256 per warp: eight lanes hold row lane / 8, lane sub = lane % 8 the
// 16-byte bf16 chunks sub + 8 k of it, x[8 k + e] = row[8 (sub + 8 k) + e].  Three of
// the eight stages of a normalised Hadamard transform cross lanes (five with a row
// to a warp), and a chunk is a whole 16-byte swizzle unit.  N = 16: the remaining
// seven stages of one half of the channels, after the stage across the halves.
template <int N>
__device__ __forceinline__ void fwht256(float (&x)[N], int sub) {
  auto in_regs = [&](int h) {
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (!(i & h)) {
        const float a = x[i], c = x[i + h];
        x[i] = a + c;
        x[i + h] = a - c;
      }
  };
  in_regs(1);
  in_regs(2);
  in_regs(4);
#pragma unroll
  for (int h = 1; h < 8; h <<= 1) {
    const float sg = (sub & h) ? -1.f : 1.f;             // a product with +-1 is exact
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const float y = __shfl_xor_sync(0xffffffffu, x[i], h);
      x[i] = fmaf(sg, x[i], y);
    }
  }
  in_regs(8);
  if constexpr (N == 32) in_regs(16);
#pragma unroll
  for (int i = 0; i < N; ++i) x[i] *= 0.0625f;           // 1 / sqrt(256)
}
// The four chunks of this lane of a bf16 row (zeros without one).
__device__ __forceinline__ void load_chunks(const __nv_bfloat16* row, int sub, uint4 (&u)[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k)
    u[k] = row ? *reinterpret_cast<const uint4*>(row + 8 * (sub + 8 * k)) : make_uint4(0, 0, 0, 0);
}
__device__ __forceinline__ void unpack_chunks(const uint4 (&u)[4], float (&x)[32]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t w[4] = {u[k].x, u[k].y, u[k].z, u[k].w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[8 * k + 2 * i] = __uint_as_float(w[i] << 16);
      x[8 * k + 2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
  }
}

__device__ __forceinline__ uint64_t fmul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// One producer thread's packed part of a tile and two of its warp's column scales.
// Keys: 64 channels of one token; values: 32 channels of two tokens.
template <int BITS, bool V>
struct Packed {
  static constexpr int NT = V ? 2 : 1, NW = V ? BITS : 2 * BITS;
  uint32_t c[NT][NW];                // codes
  uint32_t s[NT], z[NT], r[NT];      // scale, offset and row scale: fp16 bits
  __half2 col;
};
__device__ __forceinline__ float h2f(uint32_t bits) {
  return __half2float(__ushort_as_half((unsigned short)bits));
}
// A 16-bit load into a register of its own: two that the compiler packs into one
// register make the warp wait for them where they are issued.
__device__ __forceinline__ uint32_t ld16(const __half* p) {
  uint32_t v;
  asm volatile("ld.global.u16 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

template <int N>
__device__ __forceinline__ void load_words(uint32_t (&w)[N], const uint8_t* p) {
  if constexpr (N >= 4) {
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      const uint4 u = *reinterpret_cast<const uint4*>(p + 4 * i);
      w[i] = u.x; w[i + 1] = u.y; w[i + 2] = u.z; w[i + 3] = u.w;
    }
  } else {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    w[0] = u.x; w[1] = u.y;
  }
}

// Where a head's coded keys or values start.
struct Rows {
  const uint8_t* c;
  const __half *s, *z, *r, *col;
};

// The keys (this CTA's 32) or values (its half of the channels) of the tile whose
// first token is coded row q0 (-32: its second half is row 0), of `rows` coded rows.
// Lanes whose tokens are not coded load a row that is, which is not used: loads
// under a branch that divides the warp were waited for at its end (1,600 cycles a
// tile).
template <int BITS, bool V>
__device__ __forceinline__ void load_packed(const Rows& r, int q0, int rows, uint32_t rank, int w,
                                            int lane, Packed<BITS, V>& p) {
  const int ch = V ? (int)rank * (kD / 2) + w * 32 : w * 64;
#pragma unroll
  for (int u = 0; u < p.NT; ++u) {
    const int t = V ? 2 * lane + u : (int)rank * kHalf + lane;
    const int q = min(max(q0 + t, 0), rows - 1);
    load_words<p.NW>(p.c[u], r.c + ((int64_t)q * kD + ch) * BITS / 8);
    const int64_t m = (int64_t)q * (kD / kG) + ch / kG;
    p.s[u] = ld16(r.s + m);
    p.z[u] = ld16(r.z + m);
    p.r[u] = ld16(r.r + q);
  }
  // keys: 64 channels' column scales; values: 32 channels', for each half of the tile
  const int t = V ? (lane >> 4) * kHalf : (int)rank * kHalf;
  const int qc = min(max(q0 + t, 0), rows - 1) / kG;
  p.col = *reinterpret_cast<const __half2*>(r.col + (int64_t)qc * kD + ch + 2 * (V ? lane & 15 : lane));
}

// The coded keys or values of a tile into kv, for lanes whose tokens are coded
// (`in`).  col: this warp's 64 floats of shared memory.
template <int BITS, bool V>
__device__ __forceinline__ void build_coded(const Packed<BITS, V>& p, bool in, int w, int lane,
                                            float* col, unsigned char* kv) {
  __syncwarp();                                  // the previous tile's scales are read
  *reinterpret_cast<float2*>(col + 2 * lane) = __half22float2(p.col);
  __syncwarp();
  if (!in) return;
  const uint64_t bias2 = f2pack(-8388608.f, -8388608.f);
  if constexpr (!V) {
    // K: 8 chunks of 8 channels of token `lane` of the half
    const float kr = h2f(p.r[0]);
    const float ks = h2f(p.s[0]) * kr, kz = h2f(p.z[0]) * kr;
    const uint64_t ks2 = f2pack(ks, ks), kz2 = f2pack(kz, kz);
    unsigned char* kbase = kv + w * (kHalf * 128);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint32_t cw = p.c[0][c * BITS / 4] >> (c * 8 * BITS % 32);
      const float4 c0 = *reinterpret_cast<const float4*>(col + 8 * c);
      const float4 c1 = *reinterpret_cast<const float4*>(col + 8 * c + 4);
      const uint64_t cc[4] = {f2pack(c0.x, c0.y), f2pack(c0.z, c0.w), f2pack(c1.x, c1.y),
                              f2pack(c1.z, c1.w)};
      uint32_t h[4], l[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint64_t code = fadd2(f2pack(code_biased<BITS>(cw, 2 * i), code_biased<BITS>(cw, 2 * i + 1)), bias2);
        const uint64_t k2 = fmul2(ffma2(code, ks2, kz2), cc[i]);
        float a, b;
        f2unpack(k2, a, b);
        h[i] = pack_bf16(a, b);
        const float ah = __uint_as_float(h[i] << 16), bh = __uint_as_float(h[i] & 0xFFFF0000u);
        float ra, rb;
        f2unpack(fadd2(k2, f2pack(-ah, -bh)), ra, rb);
        l[i] = pack_bf16(ra, rb);
      }
      const int off = sw128(lane, c);
      *reinterpret_cast<uint4*>(kbase + kKH + off) = make_uint4(h[0], h[1], h[2], h[3]);
      *reinterpret_cast<uint4*>(kbase + kKL + off) = make_uint4(l[0], l[1], l[2], l[3]);
    }
  } else {
    // V^T: rows 32 w + e, tokens 2 lane and 2 lane + 1
    float s[2], z[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float vr = h2f(p.r[u]);
      s[u] = h2f(p.s[u]) * vr;
      z[u] = h2f(p.z[u]) * vr;
    }
    const uint64_t vs2 = f2pack(s[0], s[1]), vz2 = f2pack(z[0], z[1]);
    const float* vcol = col + (lane >> 4) * 32;
    unsigned char* vbase = kv + kVT + w * 32 * 128 + (lane & 3) * 4;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float4 c4 = *reinterpret_cast<const float4*>(vcol + 4 * c);
      const float cc[4] = {c4.x, c4.y, c4.z, c4.w};
      const uint32_t w0 = p.c[0][c * BITS / 8] >> (c * 4 * BITS % 32);
      const uint32_t w1 = p.c[1][c * BITS / 8] >> (c * 4 * BITS % 32);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int e = 4 * c + i;
        const uint64_t code = fadd2(f2pack(code_biased<BITS>(w0, i), code_biased<BITS>(w1, i)), bias2);
        float a, b;
        f2unpack(fmul2(ffma2(code, vs2, vz2), f2pack(cc[i], cc[i])), a, b);
        *reinterpret_cast<uint32_t*>(vbase + e * 128 + (((lane >> 2) ^ (e & 7)) << 4)) = pack_h2(a, b);
      }
    }
  }
}

// The full-precision tokens (sinks, staged tokens, zeros beyond T) of a tile.  Keys:
// the 32 at t0, into rows 0 .. 31 of the share.  Values: this CTA's half of the
// channels of the halves of the tile at t0 that in0, in1 do not name as coded.
// A warp takes four tokens at a time; all its rows are loaded before the first
// is rotated forward.
template <bool V>
__device__ __noinline__ void build_full(const Geom& g, int b, int h, int t0, int T, uint32_t rank,
                                        bool in0, bool in1, int w, int lane, unsigned char* kv) {
  constexpr int NW = kProdWarps / 2, NT = (V ? kTok : kHalf) / (4 * NW);
  const int sub = lane & 7;
  uint4 raw[NT][4];
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const int t = t0 + 4 * (w + NW * i) + (lane >> 3);
    const __nv_bfloat16* src = nullptr;
    if (t < T && !(i < NT / 2 || !V ? in0 : in1))
      src = t < g.S ? plane_ptr<__nv_bfloat16>(g, V ? KVQ_PLANE_V_FULL : KVQ_PLANE_K_FULL, b, h, t, 0)
                    : plane_ptr<__nv_bfloat16>(g, V ? KVQ_PLANE_V_PEND : KVQ_PLANE_K_PEND, b, h,
                                               (t - g.S) % kG, 0);
    load_chunks(src, sub, raw[i]);
  }
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    if (i < NT / 2 || !V ? in0 : in1) continue;
    const int r = 4 * (w + NW * i) + (lane >> 3);
    float x[32];
    unpack_chunks(raw[i], x);
    if constexpr (!V) {
      fwht256(x, sub);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint32_t hw[4], lw[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float x0 = x[8 * k + 2 * e], x1 = x[8 * k + 2 * e + 1];
          hw[e] = pack_bf16(x0, x1);
          lw[e] = pack_bf16(x0 - __uint_as_float(hw[e] << 16), x1 - __uint_as_float(hw[e] & 0xFFFF0000u));
        }
        unsigned char* d = kv + k * (kHalf * 128) + sw128(r, sub);
        *reinterpret_cast<uint4*>(d + kKH) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
        *reinterpret_cast<uint4*>(d + kKL) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
      }
    } else {
      // the stage across the channel halves, then the half that is this CTA's
      const float sg = rank ? -1.f : 1.f;
      float y[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) y[e] = fmaf(sg, x[16 + e], x[e]);
      fwht256(y, sub);
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int e = 0; e < 8; ++e)
          *reinterpret_cast<__half*>(kv + kVT + sw128(8 * (sub + 8 * k) + e, r >> 3) + (r & 7) * 2) =
              __float2half_rn(y[8 * k + e]);
    }
  }
}

// The tile loop of the warps that build keys (V false) or values.
template <int BITS, bool V>
__device__ __forceinline__ void produce(const Geom& g, int b, int h, int T, int ntiles, uint32_t rank,
                                        int w, int lane, float* col, unsigned char* kv_base,
                                        uint64_t* kv_full, uint64_t* kv_free, volatile int* abort) {
  // S and the coded tokens are multiples of 32, so 32 tokens are either all
  // coded, inside one block's column scales, or all full precision
  const int nbq = kvarn_nblocks(T, g.S, kG) * kG;
  auto coded = [&](int t0) { return t0 >= g.S && t0 < g.S + nbq; };
  Rows rows = {};
  if (nbq > 0) {
    rows.c = plane_ptr<uint8_t>(g, V ? KVQ_PLANE_V_CODES : KVQ_PLANE_K_CODES, b, h, 0);
    rows.s = plane_ptr<__half>(g, V ? KVQ_PLANE_V_SCALE : KVQ_PLANE_K_SCALE, b, h, 0);
    rows.z = plane_ptr<__half>(g, V ? KVQ_PLANE_V_ZERO : KVQ_PLANE_K_ZERO, b, h, 0);
    rows.r = plane_ptr<__half>(g, V ? KVQ_PLANE_V_ROW : KVQ_PLANE_K_ROW, b, h, 0);
    rows.col = plane_ptr<__half>(g, V ? KVQ_PLANE_V_COL : KVQ_PLANE_K_COL, b, h, 0);
  }
  Packed<BITS, V> cur = {}, nxt = {};
  if (coded(0) || coded(kHalf)) load_packed<BITS, V>(rows, 0 - g.S, nbq, rank, w, lane, nxt);
  for (int j = 0; j < ntiles; ++j) {
    const int t0 = j * kTok, t1 = t0 + kTok, kb = j % kKvBufs;
    cur = nxt;
    if (j + 1 < ntiles && (coded(t1) || coded(t1 + kHalf)))
      load_packed<BITS, V>(rows, t1 - g.S, nbq, rank, w, lane, nxt);
    const bool ok = j < kKvBufs || mbar_wait_or_abort(&kv_free[kb], ((j - kKvBufs) / kKvBufs) & 1, abort);
    if (!__all_sync(0xffffffffu, ok)) break;
    unsigned char* kv = kv_base + kb * kKvB;
    const bool in0 = coded(V ? t0 : t0 + (int)rank * kHalf), in1 = V ? coded(t0 + kHalf) : in0;
    if (in0 || in1) build_coded<BITS, V>(cur, V && lane >= 16 ? in1 : in0, w, lane, col, kv);
    if (!in0 || !in1)
      build_full<V>(g, b, h, V ? t0 : t0 + (int)rank * kHalf, T, rank, in0, in1, w, lane, kv);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // for the MMAs' reads
    __syncwarp();
    if (lane == 0) mbar_arrive_pair(mapa(&kv_full[kb], 0));
  }
}

template <int KB, int VB>
__global__ void __launch_bounds__(kThreads, 1)
attend_prefill_kvarn_kernel(Geom g, const __nv_bfloat16* __restrict__ q, int L, float scale,
                            __nv_bfloat16* __restrict__ out, int nq, int* err) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t kv_full[kKvBufs], kv_free[kKvBufs], s_full[kSBufs], p_full[kSBufs],
      s_free[kSBufs], done_bar;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int qpair = (gridDim.x - 1 - blockIdx.x) / 2;  // longest first
  const int hkv = blockIdx.y, b = blockIdx.z;
  const int grp = g.Hq / g.H;
  const int T = cache_tokens(g);
  const int q0 = (2 * qpair + (int)rank) * nq;
  const int nql = min(nq, L - q0);                     // <= 0: no query here, only a share of K/V
  const int pos_first = T - L + q0;
  const int t_end = T - L + min((2 * qpair + 2) * nq, L);   // the pair's keys [0, t_end)
  const int ntiles = (t_end + kTok - 1) / kTok;
  volatile int* abort = &abort_flag;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kKvBufs; ++i) {
      mbar_init(&kv_full[i], 2 * kProdWarps);
      mbar_init(&kv_free[i], 1);
    }
    for (int i = 0; i < kSBufs; ++i) {
      mbar_init(&s_full[i], 1);
      mbar_init(&p_full[i], 2 * (kM / 32));
      mbar_init(&s_free[i], 1);
    }
    mbar_init(&done_bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 12) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;"
                 ::"r"(smem_u32(&tmem_base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  // rotate the query rows, four to a warp: the high part into the swizzled Q tile,
  // the bf16 remainder into a staging row (then TMEM)
  const int sub = lane & 7;
  constexpr int kPasses = (kM / 4 + kThreads / 32 - 1) / (kThreads / 32);
  {
    uint4 raw[kPasses][4];
#pragma unroll
    for (int i = 0; i < kPasses; ++i) {
      const int r = 4 * (warp + i * (kThreads / 32)) + (lane >> 3), hl = r / nq, qi = r % nq;
      load_chunks(r < kM && hl < grp && qi < nql
                      ? q + (((int64_t)b * g.Hq + hkv * grp + hl) * L + q0 + qi) * kD
                      : nullptr,
                  sub, raw[i]);
    }
#pragma unroll
    for (int i = 0; i < kPasses; ++i) {
      const int r = 4 * (warp + i * (kThreads / 32)) + (lane >> 3);
      if (r >= kM) break;                              // the whole warp: kM is a multiple of 4
      float x[32];
      unpack_chunks(raw[i], x);
      fwht256(x, sub);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint32_t hw[4], lw[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float x0 = x[8 * k + 2 * e], x1 = x[8 * k + 2 * e + 1];
          hw[e] = pack_bf16(x0, x1);
          lw[e] = pack_bf16(x0 - __uint_as_float(hw[e] << 16), x1 - __uint_as_float(hw[e] & 0xFFFF0000u));
        }
        *reinterpret_cast<uint4*>(smem + kQOff + k * (kM * 128) + sw128(r, sub)) =
            make_uint4(hw[0], hw[1], hw[2], hw[3]);
        *reinterpret_cast<uint4*>(smem + kKvOff + r * kQlPitch + 16 * (sub + 8 * k)) =
            make_uint4(lw[0], lw[1], lw[2], lw[3]);
      }
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  if (warp < 4) {
    const unsigned char* src = smem + kKvOff + threadIdx.x * kQlPitch;
#pragma unroll 2
    for (int c = 0; c < 128; c += 16) {
      uint32_t v[16];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint4 u = *reinterpret_cast<const uint4*>(src + 4 * c + 16 * i);
        v[4 * i] = u.x; v[4 * i + 1] = u.y; v[4 * i + 2] = u.z; v[4 * i + 3] = u.w;
      }
      tmem_st16(tmem + lane_base + kTmQ + c, v);
    }
    tmem_wait_st();
  }
  tc_fence_before();
  __syncthreads();                                     // Q_lo in TMEM, the K/V area is free
  cluster_sync();                                      // in both CTAs, and their barriers are set up
  tc_fence_after();

  float inv_l = 0.f;
  if (warp >= 4 && warp < 12) {
    // ---------------- producers: reconstruct K and V tiles ----------------
    const int pw = warp - 4;
    float* col = reinterpret_cast<float*>(smem + kColOff) + pw * 64;
    if (pw < kProdWarps / 2)
      produce<KB, false>(g, b, hkv, T, ntiles, rank, pw, lane, col, smem + kKvOff, kv_full, kv_free, abort);
    else
      produce<VB, true>(g, b, hkv, T, ntiles, rank, pw - kProdWarps / 2, lane, col, smem + kKvOff, kv_full,
                        kv_free, abort);
  } else if (warp == 12) {
    if (rank == 0) {
      // ---------------- MMA issuer ----------------
      // Q K^T of tile j + 1, then P V of tile j, each blocking on what it needs (a
      // loop that polled for whichever came first answered later: 898 us for 8192
      // tokens, 855 with a warp for each product, 824 so).  The whole warp runs
      // the loop and one elected lane issues.  A K step of 16 elements advances a
      // descriptor by 32 bytes.
      constexpr uint32_t id_qk = idesc_bf16(2 * kM, kTok);
      constexpr uint32_t id_pv = idesc_f16(2 * kM, kD);
      const uint64_t qdesc0 = sw128_desc(smem + kQOff);
      const uint64_t kdesc0 = sw128_desc(smem + kKvOff);
      const uint64_t vdesc0 = sw128_desc(smem + kKvOff + kVT);
      const bool leader = elect_one();
      bool ok = true;
      for (int i = 0; i <= ntiles; ++i) {
        if (i < ntiles) {
          const int j = i, kb = j % kKvBufs, sb = j % kSBufs;
          ok = warp_wait(&kv_full[kb], (j / kKvBufs) & 1, abort) &&
               (j < kSBufs || warp_wait(&s_free[sb], ((j - kSBufs) / kSBufs) & 1, abort));
          if (!ok) break;
          tc_fence_after();
          if (leader) {
            const uint32_t ts = tmem + kTmS + sb * kTok;
#pragma unroll
            for (int kk = 0; kk < kD / 16; ++kk) {
              // Q atom: 128 rows x 128 B (1024 units); K atom: 32 rows x 128 B (256 units)
              const uint64_t qd = qdesc0 + (uint64_t)((kk >> 2) * 1024 + (kk & 3) * 2);
              const uint64_t kd = kdesc0 + (uint64_t)(kb * (kKvB >> 4) + (kk >> 2) * 256 + (kk & 3) * 2);
              umma_pair_a_fill(ts, qd, kd + (kKH >> 4), id_qk, kk > 0);     // Q_hi read once
              umma_pair_a_lastuse(ts, qd, kd + (kKL >> 4), id_qk, 1);       // for K hi and lo
              umma_pair_ts(ts, tmem + kTmQ + kk * 8, kd + (kKH >> 4), id_qk, 1);
            }
            umma_commit_pair(&s_full[sb]);
          }
          __syncwarp();
        }
        if (i > 0) {
          const int j = i - 1, kb = j % kKvBufs, sb = j % kSBufs;
          ok = warp_wait(&p_full[sb], (j / kSBufs) & 1, abort);
          if (!ok) break;
          tc_fence_after();
          if (leader) {
            const uint32_t tp = tmem + kTmS + sb * kTok;               // P (fp16 pairs) over S
#pragma unroll
            for (int kk = 0; kk < kTok / 16; ++kk)
              umma_pair_ts(tmem + kTmO, tp + kk * 8, vdesc0 + (uint64_t)(kb * (kKvB >> 4) + kk * 2), id_pv,
                           (j > 0 || kk > 0) ? 1u : 0u);
            umma_commit_pair(&s_free[sb]);            // S/P buffer free, and O holds tile j
            umma_commit_pair(&kv_free[kb]);
          }
          __syncwarp();
        }
      }
      if (leader) umma_commit_pair(&done_bar);   // every MMA issued above has completed
      if (lane == 0 && !mbar_wait(&done_bar, 0)) *abort = 1;
      __syncwarp();
    }
  } else {
    // ---------------- softmax: one row per thread ----------------
    const int row = threadIdx.x;
    const int hl = row / nq, qi = row % nq;
    const int pos = hl < grp && qi < nql ? pos_first + qi : -1;
    const uint32_t s_col = tmem + lane_base + kTmS, o_col = tmem + lane_base + kTmO;
    const float c2 = scale * 1.4426950408889634f;   // scores in log2 units
    const uint64_t c22 = f2pack(c2, c2);
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int j = 0; j < ntiles; ++j) {
      const int sb = j % kSBufs, t0 = j * kTok;
      // the second CTA first for the P V that freed this buffer, so that the waits on s_free
      // below skip none of its phases (a parity tells a phase only from its neighbours);
      // the first CTA's issuer saw that phase end before it issued these scores, but that
      // the second hears of it before it hears of them is not given
      if ((rank == 1 && j >= kSBufs && !warp_wait(&s_free[sb], ((j - kSBufs) / kSBufs) & 1, abort)) ||
          !warp_wait(&s_full[sb], (j / kSBufs) & 1, abort)) {
        ok = false;
        break;
      }
      tc_fence_after();
      uint32_t sr[kTok];
#pragma unroll
      for (int c = 0; c < kTok; c += 16) tmem_ld16_nowait(s_col + sb * kTok + c, sr + c);
      tmem_wait_ld();
      if (t0 + kTok - 1 > pos) {               // some key of the tile is in the row's future
#pragma unroll
        for (int i = 0; i < kTok; ++i)
          if (t0 + i > pos) sr[i] = __float_as_uint(-INFINITY);
      }
      float mx4[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const uint32_t* v = sr + 16 * a;
        float mv = fmax3(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]));
#pragma unroll
        for (int k = 3; k < 15; k += 2) mv = fmax3(mv, __uint_as_float(v[k]), __uint_as_float(v[k + 1]));
        mx4[a] = fmaxf(mv, __uint_as_float(v[15]));
      }
      const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      const float m_new = fmaxf(m, mx * c2);   // (c2 > 0: the maximum commutes)
      if (j == 0) {
        m = m_new;
      } else if (__any_sync(0xffffffffu, m_new > m + kRescale)) {
        // O is rewritten: the P V of tile j - 1 must have completed
        if (!warp_wait(&s_free[(j - 1) % kSBufs], ((j - 1) / kSBufs) & 1, abort)) {
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
        for (int c = 0; c < kD; c += 16) {
          uint32_t o[16];
          tmem_ld16_nowait(o_col + c, o);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
          tmem_st16(o_col + c, o);
        }
      }
      // P = 2^(s c2 - m) as fp16 pairs over the first 32 columns of this S
      // buffer (a row without any visible key so far has m = -inf and P = 0)
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
      tmem_st16(s_col + sb * kTok, pk);
      tmem_st16(s_col + sb * kTok + 16, pk + 16);
      float s0, s1;
      f2unpack(sum2, s0, s1);
      l += s0 + s1;
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_pair(mapa(&p_full[sb], 0));
    }
    if (ok && ntiles > 0 &&
        !warp_wait(&s_free[(ntiles - 1) % kSBufs], ((ntiles - 1) / kSBufs) & 1, abort))
      ok = false;
    tc_fence_after();
    inv_l = ok && l > 0.f ? 1.f / l : 0.f;
  }
  // ---------------- epilogue: normalise, rotate back, store ----------------
  tc_fence_before();
  __syncthreads();                                     // every MMA has completed
  tc_fence_after();
  const bool good = !*abort;
  float* os = reinterpret_cast<float*>(smem);
  if (warp < 4 && good) {
    float* orow = os + threadIdx.x * kOPitch;
#pragma unroll 1
    for (int c = 0; c < kD; c += 16) {
      uint32_t o[16];
      tmem_ld16_nowait(tmem + lane_base + kTmO + c, o);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 16; i += 4)
        *reinterpret_cast<float4*>(orow + c + i) =
            make_float4(__uint_as_float(o[i]) * inv_l, __uint_as_float(o[i + 1]) * inv_l,
                        __uint_as_float(o[i + 2]) * inv_l, __uint_as_float(o[i + 3]) * inv_l);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (good) {
    for (int r = 4 * warp + (lane >> 3); r < kM; r += 4 * (kThreads / 32)) {
      const int hl = r / nq, qi = r % nq;
      float x[32];
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int e = 0; e < 8; e += 4) {
          const float4 u = *reinterpret_cast<const float4*>(os + r * kOPitch + 8 * (sub + 8 * k) + e);
          x[8 * k + e] = u.x; x[8 * k + e + 1] = u.y; x[8 * k + e + 2] = u.z; x[8 * k + e + 3] = u.w;
        }
      fwht256(x, sub);
      if (hl >= grp || qi >= nql) continue;
      __nv_bfloat16* dst = out + (((int64_t)b * g.Hq + hkv * grp + hl) * L + q0 + qi) * kD;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        *reinterpret_cast<uint4*>(dst + 8 * (sub + 8 * k)) =
            make_uint4(pack_bf16(x[8 * k], x[8 * k + 1]), pack_bf16(x[8 * k + 2], x[8 * k + 3]),
                       pack_bf16(x[8 * k + 4], x[8 * k + 5]), pack_bf16(x[8 * k + 6], x[8 * k + 7]));
    }
  }
  if (threadIdx.x == 0 && !good) atomicOr(err, 8);
  // the issuer's last arrival on this CTA's barriers has landed
  if (warp == 12 && lane == 0 && rank == 1 && !mbar_wait(&done_bar, 0)) atomicOr(err, 8);
  tc_fence_before();
  cluster_sync();                                      // neither CTA's TMEM or shared memory is in use
  if (warp == 12) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

template <int KB, int VB>
cudaError_t launch(const Geom& g, const void* q, int L, float scale, void* out, int* err,
                   cudaStream_t s) {
  auto kern = attend_prefill_kvarn_kernel<KB, VB>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kAlloc);
  if (e != cudaSuccess) return e;
  const int nq = kM / (g.Hq / g.H);
  launch_pdl_pair(kern, dim3((L + 2 * nq - 1) / (2 * nq) * 2, g.H, g.B), dim3(kThreads), (size_t)kAlloc, s, g,
             reinterpret_cast<const __nv_bfloat16*>(q), L, scale,
             reinterpret_cast<__nv_bfloat16*>(out), nq, err);
  return cudaGetLastError();
}

}  // namespace

// bf16 KVarN caches at head_dim 256 with 64-token blocks, 2- or 4-bit codes and a
// number of sinks that is a multiple of 32 (32 tokens of a tile are then either all
// coded, inside one column-scale block, or all full precision).
bool prefill_kvarn_supported(const Geom& g) {
  return g.fmt == KVQ_FMT_KVARN && g.layout == KVQ_LAYOUT_UNIFORM && g.act == KVQ_BF16 &&
         g.D == kD && g.G == kG && g.S % kHalf == 0 && (g.kb == 2 || g.kb == 4) &&
         (g.vb == 2 || g.vb == 4);
}

cudaError_t launch_prefill_kvarn(const Geom& g, const void* q, int L, float scale, void* out,
                                 int* err, cudaStream_t s) {
  if (g.kb == 4)
    return g.vb == 4 ? launch<4, 4>(g, q, L, scale, out, err, s)
                     : launch<4, 2>(g, q, L, scale, out, err, s);
  return g.vb == 4 ? launch<2, 4>(g, q, L, scale, out, err, s)
                   : launch<2, 2>(g, q, L, scale, out, err, s);
}

}  // namespace kvq
