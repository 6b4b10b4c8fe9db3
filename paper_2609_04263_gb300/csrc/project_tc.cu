// LoRA-adapted Q/K/V projection on the 5th-generation tensor cores (tcgen05),
// for many rows (prefill).  Section 3, Eq. (1) and Eq. (lora), with the
// adapter kept as an explicit rank-r branch (Section 3.4):
//   y = x W_p^T + (alpha/r) (x A_p^T) B_p^T,   then RoPE on q and k.
//
// A cluster of two CTAs computes a 256 x BN tile of y inside one projection p
// (BN holds whole heads) as one pair (cta_group::2): each CTA keeps its own 128
// rows of x, the accumulator rows that go with them and one half of the BN
// rows of W.  One warp of each CTA streams its K-slices of x, W and A_p with
// TMA (128-byte swizzle) through a kStages-deep ring whose full barriers sit in
// the first CTA; one warp of that CTA issues tcgen05.mma for the pair: x W^T
// accumulates in TMEM columns [0, BN), x A_p^T in columns [BN, BN + rank).
// Afterwards the epilogue threads (one per row / TMEM lane, the columns in two
// halves) read x A_p^T, scale it by alpha/r, round it to bf16 and write it to
// shared memory as an MMA operand; one more MMA pass adds (alpha/r)(x A_p^T) B_p^T
// into the main accumulator.  The epilogue reads the tile from TMEM, applies
// rotate-half RoPE and stores head-major [B, H, L, D].
// What bounds it: for a 256 x 256 tile of K = 4096 the main loop took 31.8 us with
// and without pairing while the issuing thread formed the shared-memory
// descriptors of every MMA; 23.5 us with descriptors formed once and constants
// added (19.2 without the x A_p^T MMAs of 16 columns, which cost the pipe as
// much as wider ones).  Each tile then waits for its epilogue: 5.7 us, 3.9 with
// the sines and cosines formed during the main loop.  8192 x 4096 -> 6144 with
// rank 16: 439 us before, 359 here (1,160 TFLOP/s).
// Every mbarrier wait is bounded; a timeout sets the library's error word and
// the CTA still frees its TMEM.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <math.h>
#include <string.h>

#include <mutex>
#include <type_traits>

#include "kvq_internal.cuh"
#include "quant_common.cuh"
#include "tc_common.cuh"

namespace kvq {

// shared with project.cu
void rope_theta_table(float rope_base, int D, float* hi, float* lo);

namespace {

constexpr int BM = 128;
constexpr int BK = 64;              // bf16 elements per 128-byte swizzle row
constexpr int kStages = 5;
constexpr int kEpiWarps = 8;       // 2 threads per row of the epilogue
// the warps that issue the loads and the MMAs: two more than the epilogue's, or
// two of them where dequantising warps (from kDqWarp0 on, the epilogue's second
// half among them) need the registers
template <bool NF4> constexpr int kTmaWarp = NF4 ? 0 : kEpiWarps;
template <bool NF4> constexpr int kMmaWarp = NF4 ? 1 : kEpiWarps + 1;
constexpr int kDqWarp0 = 4;
using namespace tc;

// The 16 NF4 levels, code 0 .. 15, as QLoRA publishes the data type.
__device__ __forceinline__ constexpr float nf4_level(int code) {
  constexpr float lv[16] = {
      -1.0f, -0.6961928009986877f, -0.5250730514526367f, -0.39491748809814453f,
      -0.28444138169288635f, -0.18477343022823334f, -0.09105003625154495f, 0.0f,
      0.07958029955625534f, 0.16093020141124725f, 0.24611230194568634f, 0.33791524171829224f,
      0.44070982933044434f, 0.5626170039176941f, 0.7229568362236023f, 1.0f};
  return lv[code];
}
// Byte permute; a selector nibble 8 + k gives the sign of byte k in every bit.
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

struct TcArgs {
  void* out[3];
  int B, L, M, D, Hq, Hkv;
  int n_off[4];                 // first output column of q, k, v; total columns
  int r[3], rp[3];              // ranks and ranks padded to 16
  int pos0;
  const int* pos_dev;
  int pos_stride;
  float alpha_over_r;
  int rope;
  int k_blocks;
  int* err;
  int pack;                     // 1: code k and v into the cache g instead of storing them
  const uint8_t* nf4_codes;     // NF4 base: codes [N][d_in / 2] (two inputs a byte, low first)
  const float* nf4_absmax;      //           and one absmax per 64 inputs of a row [N][d_in / 64]
  float* plain_out;             // plain product: fp32 [M][N] row-major, no RoPE, no adapters
  int kb_wrap;                  // > 0: K slice kb of W is slice kb % kb_wrap (W repeated along K)
  Geom g;
  float theta_hi[128], theta_lo[128];
};

__device__ __forceinline__ void rope_cs(int pos, float th_hi, float th_lo, float* c, float* s) {
  const float x = (float)pos;
  const float p = x * th_hi;
  const float e = fmaf(x, th_hi, -p) + x * th_lo;
  const float k = rintf(p * 0.15915494309189535f);
  float r = fmaf(-k, 6.28125f, p);
  r = fmaf(-k, 1.9353071795864769e-3f, r);
  r = fmaf(-k, 1.0253132e-11f, r);
  r += e;
  sincosf(r, s, c);
}

// Rotate-half pair (a, b) by the angle with cosine c and sine s.  Products
// are rounded before the fused add, so both epilogues (bf16 store, or coding
// into the cache) produce the same values bit for bit.
__device__ __forceinline__ void rope_rot(float& a, float& b, float c, float s) {
  const float a0 = a, b0 = b;
  a = fmaf(a0, c, -__fmul_rn(b0, s));
  b = fmaf(b0, c, __fmul_rn(a0, s));
}

// One token's group of 32 channels (values already rounded to bf16, as the
// unfused path stores them) coded into the cache planes: 4 x 8 codes LSB
// first, fp16 scale (and offset).
template <int BITS, bool SYM>
__device__ __forceinline__ void code_group32(const Geom& g, int cplane, int splane, int zplane,
                                             int b, int h, int t, int gi, const float v[32]) {
  float lo = v[0], hi = SYM ? fabsf(v[0]) : v[0];
#pragma unroll
  for (int i = 1; i < 32; ++i) {
    if (SYM) hi = fmaxf(hi, fabsf(v[i]));
    else { lo = fminf(lo, v[i]); hi = fmaxf(hi, v[i]); }
  }
  uint64_t w[4];
  float s = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) w[q] = quant::code8<BITS, SYM>(v + 8 * q, lo, hi, &s);
  uint8_t* crow = plane_ptr<uint8_t>(g, cplane, b, h, t) + gi * (32 * BITS / 8);
  if (BITS == 2) {
    *reinterpret_cast<uint2*>(crow) = make_uint2((uint32_t)w[0] | ((uint32_t)w[1] << 16),
                                                 (uint32_t)w[2] | ((uint32_t)w[3] << 16));
  } else if (BITS == 4) {
    *reinterpret_cast<uint4*>(crow) =
        make_uint4((uint32_t)w[0], (uint32_t)w[1], (uint32_t)w[2], (uint32_t)w[3]);
  } else {
    uint4* d = reinterpret_cast<uint4*>(crow);
    d[0] = make_uint4((uint32_t)w[0], (uint32_t)(w[0] >> 32), (uint32_t)w[1], (uint32_t)(w[1] >> 32));
    d[1] = make_uint4((uint32_t)w[2], (uint32_t)(w[2] >> 32), (uint32_t)w[3], (uint32_t)(w[3] >> 32));
  }
  *plane_ptr<__half>(g, splane, b, h, t, gi) = __float2half_rn(s);
  if (!SYM) *plane_ptr<__half>(g, zplane, b, h, t, gi) = __float2half_rn(lo + 0.0f);
}

template <int BITS, bool SYM>
__device__ __forceinline__ void code_pair(const Geom& g, int which, int b, int h, int t, int g1,
                                          int g2, const float* x1, const float* x2) {
  const int cp = which ? KVQ_PLANE_V_CODES : KVQ_PLANE_K_CODES;
  const int sp = which ? KVQ_PLANE_V_SCALE : KVQ_PLANE_K_SCALE;
  const int zp = which ? KVQ_PLANE_V_ZERO : KVQ_PLANE_K_ZERO;
  code_group32<BITS, SYM>(g, cp, sp, zp, b, h, t, g1, x1);
  code_group32<BITS, SYM>(g, cp, sp, zp, b, h, t, g2, x2);
}

template <int BN>
struct Smem {
  static constexpr int A_B = BM * BK * 2;            // 16 KB
  static constexpr int B_B = BN / 2 * BK * 2;        // this CTA's half of W's rows
  static constexpr int LA_B = 32 * BK * 2;           // LoRA A slice, half of up to 64 ranks
  static constexpr int STAGE_B = A_B + B_B + LA_B;
  static constexpr int U_OFF = kStages * STAGE_B;    // (alpha/r) x A^T as bf16 operand
  static constexpr int BP_OFF = U_OFF + BM * BK * 2; // B_p tile [BN / 2][64 ranks]
  static constexpr int TOTAL = BP_OFF + BN / 2 * BK * 2 + 1024;   // + alignment slack
};

// NF4: W arrives as 4-bit NormalFloat codes; BN threads from warp 4 on (two
// per row of this CTA's half of the tile) turn each 64-input K slice into the bf16
// tile the TMA would have landed (level x absmax in fp32, rounded once),
// 128-byte swizzled, and signal it on the first CTA's w_full; the x and A_p
// slices still come by TMA.
template <int BN, bool NF4>
__host__ __device__ constexpr int tc_threads() {
  return !NF4 ? (kEpiWarps + 2) * 32 : kDqWarp0 * 32 + BN > kEpiWarps * 32 ? kDqWarp0 * 32 + BN : kEpiWarps * 32;
}
template <int BN, bool NF4>
__global__ void __launch_bounds__(tc_threads<BN, NF4>(), 1)
project_tc_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                  const __grid_constant__ CUtensorMap tm_a0, const __grid_constant__ CUtensorMap tm_a1,
                  const __grid_constant__ CUtensorMap tm_a2, const __grid_constant__ CUtensorMap tm_b0,
                  const __grid_constant__ CUtensorMap tm_b1, const __grid_constant__ CUtensorMap tm_b2,
                  const TcArgs args) {
  constexpr int kDqWarps = BN / 32;
  pdl_wait();
  pdl_trigger();
  using S = Smem<BN>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t full_bar[kStages], empty_bar[kStages], w_full[kStages];
  __shared__ uint64_t u_bar, bp_bar, acc_bar;
  __shared__ uint32_t tmem_base;
  __shared__ int fail, peer_fail;

  bool app_ok = true;                    // appending: the cache has room for the L tokens
  const int T0 = args.pack ? append_begin(args.g, args.L, &app_ok) : 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();  // 0 issues the MMAs
  const int pair = blockIdx.x >> 1, ntiles = args.n_off[3] / BN;   // column tiles first
  const int n0 = pair % ntiles * BN, m0 = (pair / ntiles * 2 + (int)rank) * BM;
  const int proj = n0 < args.n_off[1] ? 0 : n0 < args.n_off[2] ? 1 : 2;
  const int r = args.r[proj], rp = args.rp[proj];
  const int rp32 = (rp + 31) / 32 * 32;  // x A_p^T columns of the pair's MMA (zeros beyond the rank)
  const CUtensorMap* tm_a = proj == 0 ? &tm_a0 : proj == 1 ? &tm_a1 : &tm_a2;
  const CUtensorMap* tm_b = proj == 0 ? &tm_b0 : proj == 1 ? &tm_b1 : &tm_b2;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&full_bar[i], 1);
      mbar_init(&empty_bar[i], 1);
      mbar_init(&w_full[i], 2 * kDqWarps); // NF4: one arrival per dequantising warp of the pair
    }
    mbar_init(&u_bar, 1);
    mbar_init(&bp_bar, 1);
    mbar_init(&acc_bar, 1);
    fail = peer_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp<NF4>) {   // TMEM: 512 columns (main BN + LoRA <= 64)
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;"
                 ::"r"(smem_u32(&tmem_base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();                        // both CTAs' barriers and TMEM exist
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  const uint32_t tmem_u = tmem + BN;
  const int KB = args.k_blocks;

  if (threadIdx.x == kTmaWarp<NF4> * 32) {
    // ---------------- TMA producer ----------------
    // (the first CTA's barriers expect both CTAs' bytes)
    const int nh = n0 + (int)rank * (BN / 2);          // this CTA's rows of W and B_p
    if (r > 0) {
      if (rank == 0) mbar_expect_tx(&bp_bar, 2 * (BN / 2) * BK * 2);
      tma_load_2d_pair(smem + S::BP_OFF, tm_b, 0, nh - args.n_off[proj], mapa(&bp_bar, 0));
    }
    for (int kb = 0; kb < KB; ++kb) {
      const int s = kb % kStages;
      if (kb >= kStages && !mbar_wait(&empty_bar[s], ((kb / kStages) - 1) & 1)) {
        atomicOr(&fail, 1);
        break;
      }
      unsigned char* st = smem + s * S::STAGE_B;
      if (rank == 0)
        mbar_expect_tx(&full_bar[s], 2 * (S::A_B + (NF4 ? 0 : S::B_B)) + (r > 0 ? rp32 * BK * 2 : 0));
      const uint32_t fb = mapa(&full_bar[s], 0);
      tma_load_2d_pair(st, &tm_x, kb * BK, m0, fb);
      if (!NF4)
        tma_load_2d_pair(st + S::A_B, &tm_w, (args.kb_wrap ? kb % args.kb_wrap : kb) * BK, nh, fb);
      if (r > 0) tma_load_2d_pair(st + S::A_B + S::B_B, tm_a, kb * BK, (int)rank * (rp32 / 2), fb);
    }
  } else if (warp == kMmaWarp<NF4> && rank == 0) {
    // ---------------- MMA issuer ----------------
    // The whole warp runs the loop (its values stay warp-uniform) and one elected
    // lane issues.  Descriptors are formed once; a stage and a K step of 16
    // elements (32 bytes) advance their start address, in 16-byte units.
    constexpr uint32_t id_main = idesc_bf16(2 * BM, BN);
    const uint32_t id_u = idesc_bf16(2 * BM, rp32 > 0 ? rp32 : 32);
    const uint64_t desc0 = sw128_desc(smem);
    const bool leader = elect_one();
    bool ok = true;
    int s = 0, phase = 0;
    for (int kb = 0; kb < KB; ++kb) {
      bool ready = mbar_wait(&full_bar[s], phase);
      if (NF4) ready = ready && mbar_wait(&w_full[s], phase);
      if (!__all_sync(0xffffffffu, ready)) {
        ok = false;
        break;
      }
      tc_fence_after();
      if (leader) {
        const uint64_t ad = desc0 + (uint64_t)(s * (S::STAGE_B >> 4));
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk)
          umma_pair(tmem, ad + 2 * kk, ad + (S::A_B >> 4) + 2 * kk, id_main, (kb | kk) != 0);
        if (r > 0)
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            umma_pair(tmem_u, ad + 2 * kk, ad + ((S::A_B + S::B_B) >> 4) + 2 * kk, id_u, (kb | kk) != 0);
        umma_commit_pair(&empty_bar[s]);   // frees the stage in both CTAs when these MMAs finish
      }
      __syncwarp();
      if (++s == kStages) {
        s = 0;
        phase ^= 1;
      }
    }
    if (leader) {
      if (!ok) atomicOr(&fail, 1);
      umma_commit_pair(&u_bar);            // all main-loop MMAs done
    }
  } else if (NF4 && warp >= kDqWarp0 && warp < kDqWarp0 + kDqWarps) {
    // ---------- NF4 dequantisation: two threads per row of this CTA's half ----------
    constexpr int TPR = 2;
    constexpr int NQ = 2 / TPR;                           // 16-byte code words per thread and slice
    const int dt = threadIdx.x - kDqWarp0 * 32;               // 0 .. BN - 1
    const int n = dt / TPR, h = dt % TPR;                 // row, part of the slice
    const int nkb = args.k_blocks, nrow = n0 + (int)rank * (BN / 2) + n;
    const uint8_t* crow = args.nf4_codes + (int64_t)nrow * (nkb * 32) + h * 16;
    const float* arow = args.nf4_absmax + (int64_t)nrow * nkb;
    // Codes and absmax of the next PF K slices in registers, PF slices to a loop
    // trip: each is refilled as soon as it has been read and is not moved, as a
    // move of a value still being loaded waits for it (272 us for 2048 x 4096 ->
    // 6144 with buffers rotated each slice, 268 without; 167 with the arrival
    // below no longer waiting for the loads).
    constexpr int PF = 4;
    uint4 cq[PF][NQ];
    float am[PF];
#pragma unroll
    for (int i = 0; i < PF; ++i) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) cq[i][q] = make_uint4(0, 0, 0, 0);
      am[i] = 0.f;
    }
    auto fetch = [&](int kb, uint4 (&x)[NQ], float& xa) {
      if (kb < KB) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) x[q] = __ldg(reinterpret_cast<const uint4*>(crow + kb * 32 + 16 * q));
        xa = __ldg(arow + kb);
      }
    };
#pragma unroll
    for (int i = 0; i < PF; ++i) fetch(i, cq[i], am[i]);
    const int rsw = (n >> 3) * 1024 + (n & 7) * 128;      // the row in the swizzled tile
    bool live = true;
    for (int kb0 = 0; kb0 < KB && live; kb0 += PF)
#pragma unroll
    for (int u = 0; u < PF; ++u) {
      const int kb = kb0 + u;
      if (kb >= KB || !live) break;
      const int s = kb % kStages;
      if (kb >= kStages) {                                // lane 0 waits for the slot, then the warp
        bool ok = true;
        if (lane == 0) ok = mbar_wait(&empty_bar[s], ((kb / kStages) - 1) & 1);
        if (!__shfl_sync(0xffffffffu, ok, 0)) {
          if (lane == 0) atomicOr(&fail, 1);
          live = false;
          break;
        }
      }
      unsigned char* wt = smem + s * S::STAGE_B + S::A_B;
      uint32_t w8[4 * NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        w8[4 * q] = cq[u][q].x; w8[4 * q + 1] = cq[u][q].y;
        w8[4 * q + 2] = cq[u][q].z; w8[4 * q + 3] = cq[u][q].w;
      }
      const float a = am[u];
      fetch(kb + PF, cq[u], am[u]);
      // The 16 levels times absmax (fp32 products, rounded to bf16 once) as bytes in
      // registers, 4 codes to a byte permute: with the levels looked up in shared
      // memory and multiplied code by code a slice took 820 cycles (166 us for 2048 x 4096
      // -> 6144; 134 so).
      uint32_t tl[4], th[4];                              // low, high bytes of entries 4 k ..
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t p0 = pack_bf16(nf4_level(4 * k) * a, nf4_level(4 * k + 1) * a);
        const uint32_t p1 = pack_bf16(nf4_level(4 * k + 2) * a, nf4_level(4 * k + 3) * a);
        tl[k] = prmt(p0, p1, 0x6420u);
        th[k] = prmt(p0, p1, 0x7531u);
      }
#pragma unroll
      for (int j = 0; j < 4 * NQ; ++j) {                  // chunk c: inputs 8c .. 8c + 7
        const int c = 4 * NQ * h + j;
        const uint32_t w = w8[j], sel = w & 0x77777777u, y = w << 4;
        uint32_t o[4];
#pragma unroll
        for (int u = 0; u < 2; ++u) {                     // inputs 4u .. 4u + 3 of the chunk
          const uint32_t s4 = u ? sel >> 16 : sel;        // entry within its half of the table
          // bytes of ones where bit 3 of the code is set: the upper half
          const uint32_t m = prmt(y, w, u ? 0xFBEAu : 0xD9C8u);
          const uint32_t lo = (prmt(tl[0], tl[1], s4) & ~m) | (prmt(tl[2], tl[3], s4) & m);
          const uint32_t hi = (prmt(th[0], th[1], s4) & ~m) | (prmt(th[2], th[3], s4) & m);
          o[2 * u] = prmt(lo, hi, 0x5140u);
          o[2 * u + 1] = prmt(lo, hi, 0x7362u);
        }
        *reinterpret_cast<uint4*>(wt + rsw + ((c ^ (n & 7)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // for the MMA's reads
      __syncwarp();
      if (lane == 0) mbar_arrive_pair(mapa(&w_full[s], 0));
    }
  }
  // ---------------- (alpha/r) x A^T -> bf16 operand in shared memory ----------
  const int row = (warp & 3) * 32 + lane;      // TMEM lane = tile row
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  const int part = warp >> 2;                  // warps 0-3 and 4-7: every other column block
  const int m = m0 + row;
  const bool active = m < args.M;              // rows past M: load, do not store
  const int mm = active ? m : 0;
  const int b = mm / args.L, l = mm % args.L;
  const int D = args.D, half = D / 2;
  const bool rope = args.rope && proj < 2;
  // A head's 32-frequency blocks go to the two parts in turn (at D = 64 its heads
  // do); this thread's blocks: part, part + 2 (D = 256), part (D = 128), 0 (D = 64).
  // Their sines and cosines are formed while the main loop runs (not over an NF4
  // base, whose dequantising warps leave no registers for them).
  auto tail = [&](auto nblocks) -> bool {
  constexpr int NB = decltype(nblocks)::value;
  constexpr int NC = NF4 ? 1 : NB;             // blocks whose sines and cosines are held
  float cs[NC * 32], sn[NC * 32];
  auto angles = [&](int k, float* c, float* s) {
    const int pos = args.pos0 + pos_of(args.pos_dev, args.pos_stride, b) + l;
    const int j0 = D == 64 ? 0 : 32 * (part + 2 * k);
#pragma unroll
    for (int i = 0; i < 32; ++i) rope_cs(pos, args.theta_hi[j0 + i], args.theta_lo[j0 + i], &c[i], &s[i]);
  };
  if (!NF4 && rope && part < 2) {
#pragma unroll
    for (int k = 0; k < NB; ++k) angles(k, cs + 32 * (k % NC), sn + 32 * (k % NC));
  }
  bool u_done = true;                          // one lane per warp polls: the issuer needs the slots
  if (lane == 0) u_done = mbar_wait(&u_bar, 0);
  const bool u_ok = __syncthreads_and(u_done) != 0;   // uniform
  tc_fence_after();
  if (r > 0 && u_ok && part < 2) {
    unsigned char* us = smem + S::U_OFF;
    for (int c0 = 16 * part; c0 < rp; c0 += 32) {
      float v[16];
      tmem_ld16(tmem_u + lane_base + c0, v);
      uint32_t w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        w[i] = pack_bf16(v[2 * i] * args.alpha_over_r, v[2 * i + 1] * args.alpha_over_r);
      // two 16-byte chunks (k = c0 .. c0+7, c0+8 .. c0+15) of row `row`,
      // placed at chunk index c ^ (row % 8) of the 128-byte row
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int chunk = (c0 / 8 + h) ^ (row & 7);
        *reinterpret_cast<uint4*>(us + row * 128 + chunk * 16) =
            make_uint4(w[4 * h], w[4 * h + 1], w[4 * h + 2], w[4 * h + 3]);
      }
    }
    // ranks rp .. 63 of the operand row are never read (the MMA uses K = rp)
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (!u_ok && threadIdx.x == 0) atomicOr(&fail, 1);
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *reinterpret_cast<volatile int*>(&fail))
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(mapa(&peer_fail, rank ^ 1)), "r"(1) : "memory");
  cluster_sync();                              // both operands of the up-projection are written
  tc_fence_after();
  const bool pair_ok = !*reinterpret_cast<volatile int*>(&fail) &&
                       !*reinterpret_cast<volatile int*>(&peer_fail);
  if (threadIdx.x == kMmaWarp<NF4> * 32 && rank == 0 && pair_ok) {
    bool ok = true;
    if (r > 0) {
      ok = mbar_wait(&bp_bar, 0);
      if (ok) {
        constexpr uint32_t id_main = idesc_bf16(2 * BM, BN);
        for (int kk = 0; kk < rp / 16; ++kk)
          umma_pair(tmem, sw128_desc(smem + S::U_OFF + kk * 32),
                    sw128_desc(smem + S::BP_OFF + kk * 32), id_main, 1);
      }
    }
    if (ok) umma_commit_pair(&acc_bar);        // else both CTAs' waits below run out
  }
  // ---------------- epilogue: RoPE and head-major store ----------------
  const bool acc_wait = pair_ok && mbar_wait(&acc_bar, 0);
  const bool good = __syncthreads_and(acc_wait) != 0;
  tc_fence_after();
  if (good && part < 2) {
    const int H = proj == 0 ? args.Hq : args.Hkv;
    const int col0 = n0 - args.n_off[proj];           // first column within projection
    __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(args.out[proj]);
    if (args.plain_out) {
      // plain product: the accumulator row as fp32
      const int N = args.n_off[3];
      for (int c = 16 * part; c < BN; c += 32) {
        float v[16];
        tmem_ld16(tmem + lane_base + c, v);
        if (!active) continue;
        float4* d = reinterpret_cast<float4*>(args.plain_out + (int64_t)m * N + n0 + c);
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
      }
      return good;
    }
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      const int j = D == 64 ? 0 : 32 * (part + 2 * k);
      if (NF4 && rope) angles(k, cs, sn);
      for (int hc = D == 64 ? 64 * part : 0; hc < BN; hc += D == 64 ? 128 : D) {   // whole heads in the tile
        const int head = (col0 + hc) / D;
        float x1[32], x2[32];
        uint32_t* u1 = reinterpret_cast<uint32_t*>(x1);
        uint32_t* u2 = reinterpret_cast<uint32_t*>(x2);
        tmem_ld16_nowait(tmem + lane_base + hc + j, u1);
        tmem_ld16_nowait(tmem + lane_base + hc + j + 16, u1 + 16);
        tmem_ld16_nowait(tmem + lane_base + hc + half + j, u2);
        tmem_ld16_nowait(tmem + lane_base + hc + half + j + 16, u2 + 16);
        tmem_wait_ld();
        if (rope) {
#pragma unroll
          for (int i = 0; i < 32; ++i) rope_rot(x1[i], x2[i], cs[32 * (k % NC) + i], sn[32 * (k % NC) + i]);
        }
        if (!active) continue;
        if (args.pack && proj > 0) {
          // append: k (after RoPE) and v rounded to bf16, then coded per token
          // in groups of 32 channels straight into the cache planes
          if (!app_ok) continue;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            x1[i] = __bfloat162float(__float2bfloat16_rn(x1[i]));
            x2[i] = __bfloat162float(__float2bfloat16_rn(x2[i]));
          }
          const Geom& gg = args.g;
          const int bits = proj == 1 ? gg.kb : gg.vb, t = T0 + l;
          const int g1 = j / 32, g2 = (half + j) / 32, which = proj - 1;
          if (gg.fmt == KVQ_FMT_SYMMETRIC) {
            if (bits == 2) code_pair<2, true>(gg, which, b, head, t, g1, g2, x1, x2);
            else if (bits == 4) code_pair<4, true>(gg, which, b, head, t, g1, g2, x1, x2);
            else code_pair<8, true>(gg, which, b, head, t, g1, g2, x1, x2);
          } else {
            if (bits == 2) code_pair<2, false>(gg, which, b, head, t, g1, g2, x1, x2);
            else if (bits == 4) code_pair<4, false>(gg, which, b, head, t, g1, g2, x1, x2);
            else code_pair<8, false>(gg, which, b, head, t, g1, g2, x1, x2);
          }
        } else {
          __nv_bfloat16* orow = out + (((int64_t)b * H + head) * args.L + l) * D;
          uint4* d1 = reinterpret_cast<uint4*>(orow + j);
          uint4* d2 = reinterpret_cast<uint4*>(orow + half + j);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            d1[i] = make_uint4(pack_bf16(x1[8 * i], x1[8 * i + 1]), pack_bf16(x1[8 * i + 2], x1[8 * i + 3]),
                               pack_bf16(x1[8 * i + 4], x1[8 * i + 5]), pack_bf16(x1[8 * i + 6], x1[8 * i + 7]));
            d2[i] = make_uint4(pack_bf16(x2[8 * i], x2[8 * i + 1]), pack_bf16(x2[8 * i + 2], x2[8 * i + 3]),
                               pack_bf16(x2[8 * i + 4], x2[8 * i + 5]), pack_bf16(x2[8 * i + 6], x2[8 * i + 7]));
          }
        }
      }
    }
  }
  return good;
  };
  // (an NF4 base has heads of 64 or 128)
  const bool good = !NF4 && D == 256 ? tail(std::integral_constant<int, NF4 ? 1 : 2>())
                                     : tail(std::integral_constant<int, 1>());
  if (threadIdx.x == 0 && !good) atomicOr(args.err, 2);
  tc_fence_before();
  __syncthreads();
  cluster_sync();                              // neither CTA's shared memory or TMEM is in use
  if (warp == kMmaWarp<NF4>) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
  // appending: the last CTA to arrive advances the cache's token count
  if (args.pack) quant::append_arrive_spread(args.g.state, T0, args.L, app_ok);
}

// ---------------------------------------------------------------------------
// host: tensor maps through the driver entry point (no libcuda link)
// ---------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// 2D bf16 tensor [rows][cols] (cols contiguous), box [box_rows][64 cols],
// 128-byte swizzle; out-of-range elements read as zero.
bool make_map(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult res = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                    box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return res == CUDA_SUCCESS;
}

template <int BN, bool NF4 = false>
cudaError_t launch_bn(const CUtensorMap maps[8], const TcArgs& a, cudaStream_t s) {
  const int smem = Smem<BN>::TOTAL;
  auto kern = project_tc_kernel<BN, NF4>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int64_t ctas = 2LL * (a.n_off[3] / BN) * ((a.M + 2 * BM - 1) / (2 * BM));
  if (ctas > INT32_MAX) return cudaErrorInvalidConfiguration;
  dim3 grid((unsigned)ctas);
  launch_pdl_pair(kern, grid, dim3(tc_threads<BN, NF4>()), smem, s, maps[0], maps[1], maps[2], maps[3], maps[4], maps[5],
                                    maps[6], maps[7], a);
  return cudaGetLastError();
}

}  // namespace

// Tile width for these head counts, or 0 if the tensor-core path does not
// cover the shape (then the caller uses the SIMT kernel).
int project_tc_tile(int Hq, int Hkv, int D, int d_in) {
  if (d_in % 64) return 0;
  const int nq = Hq * D, nk = Hkv * D;
  for (int bn : {256, 128}) {
    if (bn < D) continue;
    if (nq % bn == 0 && nk % bn == 0) return bn;
  }
  return 0;
}

// NF4 base (codes, absmax) when `w` is null.
static cudaError_t launch_tc(const void* x, int B, int L, int d_in, const void* w,
                             const uint8_t* nf4_codes, const float* nf4_absmax,
                             const void* const a[3], const void* const bm[3], const int r[3],
                             float alpha_over_r, int Hq, int Hkv, int D, int pos0,
                             const int* pos_dev, float rope_base, void* const out[3], int* err,
                             cudaStream_t s, const Geom* append_to, int pos_stride) {
  const bool nf4 = w == nullptr;
  const int bn = project_tc_tile(Hq, Hkv, D, d_in);
  if (!bn) return cudaErrorNotSupported;
  TcArgs t;
  t.nf4_codes = nf4_codes;
  t.nf4_absmax = nf4_absmax;
  t.plain_out = nullptr;
  t.kb_wrap = 0;
  t.pack = append_to != nullptr;
  if (append_to) t.g = *append_to;
  else memset(&t.g, 0, sizeof t.g);
  const int M = B * L;
  for (int i = 0; i < 3; ++i) {
    t.out[i] = out[i];
    t.r[i] = r[i];
    t.rp[i] = (r[i] + 15) / 16 * 16;
  }
  t.B = B; t.L = L; t.M = M; t.D = D; t.Hq = Hq; t.Hkv = Hkv;
  t.n_off[0] = 0; t.n_off[1] = Hq * D; t.n_off[2] = (Hq + Hkv) * D; t.n_off[3] = (Hq + 2 * Hkv) * D;
  t.pos0 = pos0; t.pos_dev = pos_dev; t.pos_stride = pos_stride; t.alpha_over_r = alpha_over_r;
  t.rope = rope_base > 0.f; t.k_blocks = d_in / 64; t.err = err;
  rope_theta_table(rope_base, D, t.theta_hi, t.theta_lo);
  CUtensorMap maps[8];
  bool ok = make_map(&maps[0], x, M, d_in, BM);
  if (nf4) maps[1] = maps[0];                       // unused: any valid map
  else ok = ok && make_map(&maps[1], w, (uint64_t)t.n_off[3], d_in, bn / 2);
  const int dout[3] = {Hq * D, Hkv * D, Hkv * D};
  for (int p = 0; p < 3 && ok; ++p) {
    if (r[p] > 0) {
      ok = make_map(&maps[2 + p], a[p], r[p], d_in, (t.rp[p] + 31) / 32 * 16) &&
           make_map(&maps[5 + p], bm[p], dout[p], r[p], bn / 2);
    } else {  // unused: any valid map
      maps[2 + p] = maps[0];
      maps[5 + p] = maps[0];
    }
  }
  if (!ok) return cudaErrorInvalidValue;
  if (nf4) return bn == 256 ? launch_bn<256, true>(maps, t, s) : launch_bn<128, true>(maps, t, s);
  return bn == 256 ? launch_bn<256>(maps, t, s) : launch_bn<128>(maps, t, s);
}

cudaError_t launch_project_tc(const void* x, int B, int L, int d_in, const void* w,
                              const void* const a[3], const void* const bm[3], const int r[3],
                              float alpha_over_r, int Hq, int Hkv, int D, int pos0,
                              const int* pos_dev, float rope_base, void* const out[3], int* err,
                              cudaStream_t s, const Geom* append_to, int pos_stride) {
  if (!w) return cudaErrorInvalidValue;
  return launch_tc(x, B, L, d_in, w, nullptr, nullptr, a, bm, r, alpha_over_r, Hq, Hkv, D, pos0,
                   pos_dev, rope_base, out, err, s, append_to, pos_stride);
}

// C [M][N] fp32 = A [M][K] B^T on tcgen05, A bf16 K-major, B's rows bf16 of Kb
// elements repeated along K (K a multiple of Kb: B(k) = Bt[:, k mod Kb]).
cudaError_t launch_gemm_tc_bf16(const void* a, int M, int K, const void* bt, int N, int Kb,
                                float* c, int* err, cudaStream_t s) {
  if (M <= 0 || N <= 0 || K <= 0 || K % 64 || Kb % 64 || K % Kb) return cudaErrorInvalidValue;
  const int bn = N % 256 == 0 ? 256 : N % 128 == 0 ? 128 : 0;
  if (!bn) return cudaErrorNotSupported;
  TcArgs t;
  memset(&t, 0, sizeof t);
  t.B = 1; t.L = M; t.M = M; t.D = 64; t.Hq = N / 64; t.Hkv = 1;
  t.n_off[0] = 0; t.n_off[1] = N; t.n_off[2] = N; t.n_off[3] = N;
  t.k_blocks = K / 64; t.kb_wrap = Kb / 64 == K / 64 ? 0 : Kb / 64; t.err = err;
  t.plain_out = c;
  CUtensorMap maps[8];
  if (!make_map(&maps[0], a, M, K, BM) || !make_map(&maps[1], bt, N, Kb, bn / 2))
    return cudaErrorInvalidValue;
  for (int i = 2; i < 8; ++i) maps[i] = maps[0];   // unused: no adapters
  return bn == 256 ? launch_bn<256>(maps, t, s) : launch_bn<128>(maps, t, s);
}

bool project_tc_nf4_supported(int Hq, int Hkv, int D, int d_in) {
  return project_tc_tile(Hq, Hkv, D, d_in) != 0;
}

cudaError_t launch_project_tc_nf4(const void* x, int B, int L, int d_in, const void* codes,
                                  const void* absmax, const void* const a[3],
                                  const void* const bm[3], const int r[3], float alpha_over_r,
                                  int Hq, int Hkv, int D, int pos0, const int* pos_dev,
                                  float rope_base, void* const out[3], int* err, cudaStream_t s,
                                  int pos_stride) {
  return launch_tc(x, B, L, d_in, nullptr, static_cast<const uint8_t*>(codes),
                   static_cast<const float*>(absmax), a, bm, r, alpha_over_r, Hq, Hkv, D, pos0,
                   pos_dev, rope_base, out, err, s, nullptr, pos_stride);
}

}  // namespace kvq
