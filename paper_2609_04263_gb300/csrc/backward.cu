// Backward of the packed path under the straight-through estimator
// (Section 3.3).  Newly appended states enter attention as
// x_hat + x - stopgrad(x): the forward sees the stored reconstruction and
// the gradient that reaches the keys and values, and through them the K and
// V adapters, is the gradient at the reconstruction, passed on unchanged.
// This is what lets the adapters train against the coded cache they will be
// served with (Sections 3.2-3.4).
//
// Attention, per (sequence, kv head) pair with its g = Hq / Hkv query heads
// stacked as M = g L rows (row m: head m / L, query m % L at position
// T - L + m % L):
//   S  = Q K^T                     P  = causal softmax(scale S) per row
//   dP = dO V^T                    dS = P o (dP - rowsum(P o dP)) scale
//   dQ = dS K                      dK = dS^T Q             dV = P^T dO
// K and V are the cache's reconstruction, materialised in fp32 in the
// caller's workspace with S (then P) and dP (then dS).
//
// Adapters (Eq. (1), Eq. (lora)): y_p = x W_p^T + (alpha/r) (x A_p^T) B_p^T,
// then RoPE on q and k.  With g_p the gradient of y_p (the output gradient
// rotated back), U_p = x A_p^T and V_p = g_p B_p:
//   dB_p = (alpha/r) g_p^T U_p      dA_p = (alpha/r) V_p^T x
//   dx   = g W + sum_p (alpha/r) V_p A_p
//
// Every product runs on one GEMM kernel with strided operands, batched over
// pairs and split over K where K is long and the output small: fp32 operands as
// three bf16 parts on the tensor cores (about 24 bits), bf16 operands as they are.
#include <math.h>

#include <type_traits>

#include "kvq_internal.cuh"
#include "proj_decode.cuh"
#include "reconstruct.cuh"

namespace kvq {
namespace {

// ---------------------------------------------------------------------------
// C[z] = alpha A[z] B[z] (+ C[z]) in fp32, A(m, k) and B(k, n) at strides.
//
// An fp32 operand x is split into three bf16 parts x = x0 + x1 + x2 (each the
// rounding of what the parts before it leave: 24 significant bits) and the
// products of parts i, j with i + j <= 2 run as mma.sync (6 of them for two
// fp32 operands, 3 when the other is bf16, 1 when both are); the dropped ones
// lie below 2^-24 of the product.  The tensor cores truncate as they
// accumulate, so they sum 16 k at a time from zero (the products of the leading
// parts last), added to the fp32 accumulator with a rounding addition: the error against
// 64 bits is not above that of the fp32 chain this replaces.  An infinite value has
// no such parts (infinity times the other operand's zero parts is NaN): a 32-k step with
// one runs in fp32 (out of line: unrolled in the loop it cost registers and 2 %).
// What bounds it is the splitting and the fragment loads, not the MMAs (about 200
// of 400 issue slots per warp and chunk at six products), which is why 64 x 64 tiles on
// mma.sync, three or four CTAs per SM and no staging in tensor memory serve here.
// All products of the attention backward of 1000 tokens, 32 / 8 heads of 128:
// 1317 us in fp32 FMA, 488 us so.
// ---------------------------------------------------------------------------
constexpr int kBM = 64, kBN = 64, kBK = 32, kGemmThreads = 128;

enum MaskMode {
  kMaskNone = 0,
  kMaskRowsQueriesColsKeys = 1,   // m: stacked query rows, n: keys (S, dP)
  kMaskRowsQueriesKKeys = 2,      // m: stacked query rows, k: keys (dQ)
  kMaskRowsKeysKQueries = 3,      // m: keys, k: stacked query rows (dK, dV)
};

struct GemmOp {
  const void* a;
  const void* b;
  float* c;
  int M, N, K;
  int64_t lda, ldb, ldc;      // A(m,k) = a[m lda + k] (K-major) or a[k lda + m]
};
struct GemmArgs {
  GemmOp op[3];               // products of one launch, alike but for pointers and sizes
  int ops;
  int64_t sa, sb, sc;         // batch strides in elements
  int batch, splits;          // grid.z = ops x batch x splits; splits > 1 adds atomically
  float alpha;
  int accumulate;             // 1: C += alpha A B (splits > 1 implies it)
  int mask, L, T;             // causal structure of the attention products
};

// Latest key position visible to any of the stacked query rows [r0, r1).
__device__ __forceinline__ int max_visible(int r0, int r1, int L, int T) {
  const int last = r1 - 1;
  if (last / L != r0 / L) return T - 1;
  return T - L + last % L;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)));
}
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One operand tile (64 rows x 32 k) in shared memory, PARTS bf16 parts of it:
// [row][k] when the operand is K-major in memory, else [k][row] (ldmatrix
// transposes); rows of 80 or 144 bytes put 8 rows in distinct banks.
template <typename E, bool KMAJOR>
struct Operand {
  static constexpr int PARTS = sizeof(E) == 4 ? 3 : 1;
  static constexpr int PITCH = KMAJOR ? kBK + 8 : kBM + 8;
  static constexpr int PART = KMAJOR ? kBM * PITCH : kBK * PITCH;   // elements
  using V4 = typename std::conditional<sizeof(E) == 4, float4, uint2>::type;   // 4 elements

  // Elements (r, k .. k + 3) or (r .. r + 3, k): four per thread and step,
  // neighbouring threads on neighbouring addresses.
  static __device__ __forceinline__ void where(int i, int* r, int* k) {
    const int idx = threadIdx.x + kGemmThreads * i;
    if (KMAJOR) { *r = idx >> 3; *k = (idx & 7) * 4; }
    else { *r = (idx & 15) * 4; *k = idx >> 4; }
  }
  // vec: rows start on 4-element boundaries.
  static __device__ __forceinline__ void load(const E* p, int64_t ld, int r0, int R, int k0, int K,
                                              bool vec, V4 (&v)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int r, k;
      where(i, &r, &k);
      r += r0;
      k += k0;
      const E* q = p + (KMAJOR ? (int64_t)r * ld + k : (int64_t)k * ld + r);
      const int left = KMAJOR ? (r < R ? K - k : 0) : (k < K ? R - r : 0);   // elements from here on
      if (vec && left >= 4) {
        v[i] = *reinterpret_cast<const V4*>(q);
      } else {
        __align__(16) E e[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) e[j] = j < left ? q[j] : E(0.f);
        v[i] = *reinterpret_cast<const V4*>(e);
      }
    }
  }
  // True if a value has no parts: infinite, NaN, or beyond bf16's range.  (Its first
  // part is then infinite or NaN and the others NaN.)
  static __device__ __forceinline__ bool store(__nv_bfloat16* s, const V4 (&v)[4]) {
    uint32_t top = 0;                // largest of the parts that are NaN (0x7FFF) in that case, as int16 pairs
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int r, k;
      where(i, &r, &k);
      __nv_bfloat16* d = s + (KMAJOR ? r * PITCH + k : k * PITCH + r);
      if constexpr (PARTS == 1) {
        *reinterpret_cast<uint2*>(d) = v[i];
        top = __vmaxs2(top, __vmaxs2(v[i].x & 0x7FFF7FFFu, v[i].y & 0x7FFF7FFFu));
      } else {
        float x[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
        for (int part = 0; part < 3; ++part) {
          uint2 u;
          uint32_t* w = &u.x;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const __nv_bfloat162 t = __floats2bfloat162_rn(x[2 * h], x[2 * h + 1]);
            w[h] = *reinterpret_cast<const uint32_t*>(&t);
            const float2 f = __bfloat1622float2(t);
            x[2 * h] -= f.x;
            x[2 * h + 1] -= f.y;
          }
          *reinterpret_cast<uint2*>(d + part * PART) = u;
          if (part == 2) top = __vmaxs2(top, __vmaxs2(u.x, u.y));
        }
      }
    }
    constexpr uint32_t kInf = 0x7F80u;
    return (top & 0xFFFFu) >= kInf || (top >> 16) >= kInf;
  }
  // Element (r, k) of a stored tile.
  static __device__ __forceinline__ float at(const __nv_bfloat16* s, int r, int k) {
    const __nv_bfloat16* p = s + (KMAJOR ? r * PITCH + k : k * PITCH + r);
    const float x = __bfloat162float(p[0]);
    if (PARTS == 1) return x;
    const float lo = __bfloat162float(p[PART]) + __bfloat162float(p[(PARTS - 1) * PART]);
    return isnan(lo) ? x : x + lo;
  }
  // The 16 x 16 A fragment at rows r, k-step k.
  static __device__ __forceinline__ void frag_a(const __nv_bfloat16* s, int r, int k, int lane,
                                                uint32_t (&f)[4]) {
    if (KMAJOR) ldsm4(f, s + (r + (lane & 15)) * PITCH + k + (lane >> 4) * 8);
    else ldsm4_t(f, s + (k + (lane >> 4) * 8 + (lane & 7)) * PITCH + r + ((lane >> 3) & 1) * 8);
  }
  // Two 16 x 8 B fragments (f[0..1], f[2..3]) at columns r, k-step k.
  static __device__ __forceinline__ void frag_b(const __nv_bfloat16* s, int r, int k, int lane,
                                                uint32_t (&f)[4]) {
    const int j = lane >> 3, i = lane & 7;
    if (KMAJOR) ldsm4(f, s + (r + (j >> 1) * 8 + i) * PITCH + k + (j & 1) * 8);
    else ldsm4_t(f, s + (k + (j & 1) * 8 + i) * PITCH + r + (j >> 1) * 8);
  }
};

// One 32-k step in fp32 into a thread's sums t[16 m + 4 n + i] (out of line: rare).
template <typename OA, typename OB>
__device__ __noinline__ void fp32_step(const __nv_bfloat16* As, const __nv_bfloat16* Bs, int row,
                                       int col, float* t) {
#pragma unroll 1
  for (int j = 0; j < 32; ++j) {
    const int r = row + 16 * (j >> 4) + 8 * ((j >> 1) & 1), c = col + 8 * ((j >> 2) & 3) + (j & 1);
    float s = t[j];
#pragma unroll 1
    for (int k = 0; k < kBK; ++k) s = fmaf(OA::at(As, r, k), OB::at(Bs, c, k), s);
    t[j] = s;
  }
}

// A_KMAJOR: A(m, k) = a[m lda + k], else a[k lda + m].
// B_KMAJOR: B(k, n) = b[n ldb + k], else b[k ldb + n].
// CHAIN: the ops are one product, their K ranges behind one another (one batch entry,
// no splits, no mask).
template <typename TA, typename TB, bool A_KMAJOR, bool B_KMAJOR, bool CHAIN>
__global__ void __launch_bounds__(kGemmThreads) bgemm_kernel(const __grid_constant__ GemmArgs g) {
  pdl_wait();
  pdl_trigger();
  using OA = Operand<TA, A_KMAJOR>;
  using OB = Operand<TB, B_KMAJOR>;
  constexpr int PA = OA::PARTS, PB = OB::PARTS;
  constexpr int kStage = PA * OA::PART + PB * OB::PART;
  extern __shared__ __align__(16) __nv_bfloat16 tiles[];          // two stages of A, B parts
  const int sp = blockIdx.z % g.splits, bz = blockIdx.z / g.splits % g.batch;
  const GemmOp op = g.op[CHAIN ? 0 : blockIdx.z / (g.splits * g.batch)];
  const TA* A = reinterpret_cast<const TA*>(op.a) + (int64_t)bz * g.sa;
  const TB* Bp = reinterpret_cast<const TB*>(op.b) + (int64_t)bz * g.sb;
  float* C = op.c + (int64_t)bz * g.sc;
  const int m0 = blockIdx.y * kBM, n0 = blockIdx.x * kBN;
  if (m0 >= op.M || n0 >= op.N) return;

  // K range of this split, clipped by the causal structure.
  int kend = op.K;
  if (g.mask == kMaskRowsQueriesColsKeys &&
      n0 > max_visible(m0, min(m0 + kBM, op.M), g.L, g.T))
    return;                                    // every score of the tile is masked
  if (g.mask == kMaskRowsQueriesKKeys) kend = min(kend, max_visible(m0, min(m0 + kBM, op.M), g.L, g.T) + 1);
  int ktiles = (kend + kBK - 1) / kBK;
  if (CHAIN)
    for (int i = 1; i < g.ops; ++i) ktiles += (g.op[i].K + kBK - 1) / kBK;
  const int per = (ktiles + g.splits - 1) / g.splits;
  const int kt0 = sp * per, kt1 = min(ktiles, kt0 + per);
  if (kt0 >= kt1 && g.splits > 1) return;

  auto aligned = [](const void* p, int64_t ld, int elem, int n) {   // rows start on n-byte boundaries
    return ((reinterpret_cast<uintptr_t>(p) | (uintptr_t)(ld * elem)) & (n - 1)) == 0;
  };
  const bool veca = aligned(A, op.lda, sizeof(TA), sizeof(typename OA::V4));
  const bool vecb = aligned(Bp, op.ldb, sizeof(TB), sizeof(typename OB::V4));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;          // this warp's 32 x 32 outputs
  float acc[2][4][4] = {};
  typename OA::V4 ra[4];
  typename OB::V4 rb[4];
  auto skip = [&](int kt) {
    return g.mask == kMaskRowsKeysKQueries &&
           max_visible(kt * kBK, min(kt * kBK + kBK, op.K), g.L, g.T) < m0;
  };
  auto load = [&](int kt) {
    if constexpr (CHAIN) {
      int i = 0;
      for (int n; kt >= (n = (g.op[i].K + kBK - 1) / kBK); ++i) kt -= n;
      const GemmOp& o = g.op[i];
      OA::load(reinterpret_cast<const TA*>(o.a), o.lda, m0, op.M, kt * kBK, o.K,
               aligned(o.a, o.lda, sizeof(TA), sizeof(typename OA::V4)), ra);
      OB::load(reinterpret_cast<const TB*>(o.b), o.ldb, n0, op.N, kt * kBK, o.K,
               aligned(o.b, o.ldb, sizeof(TB), sizeof(typename OB::V4)), rb);
    } else {
      OA::load(A, op.lda, m0, op.M, kt * kBK, kend, veca, ra);
      OB::load(Bp, op.ldb, n0, op.N, kt * kBK, kend, vecb, rb);
    }
  };
  int kt = kt0;
  while (kt < kt1 && skip(kt)) ++kt;
  if (kt < kt1) load(kt);
  int buf = 0;
  while (kt < kt1) {
    __nv_bfloat16* As = tiles + buf * kStage;
    __nv_bfloat16* Bs = As + PA * OA::PART;
    bool odd = OA::store(As, ra);
    odd |= OB::store(Bs, rb);
    // (two bf16 operands multiply as they are)
    if (PA + PB > 2) odd = __syncthreads_or(odd);
    else __syncthreads();
    int nxt = kt + 1;
    while (nxt < kt1 && skip(nxt)) ++nxt;
    if (nxt < kt1) load(nxt);                  // prefetch the next tile into registers
    if (PA + PB > 2 && odd) {                  // a value without parts: in fp32
      float t[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) t[i] = acc[i >> 4][(i >> 2) & 3][i & 3];
      fp32_step<OA, OB>(As, Bs, wm + (lane >> 2), wn + 2 * (lane & 3), t);
#pragma unroll
      for (int i = 0; i < 32; ++i) acc[i >> 4][(i >> 2) & 3][i & 3] = t[i];
    } else
#pragma unroll
    for (int ks = 0; ks < kBK; ks += 16) {
      float c[2][4][4] = {};                   // this step's sums
      uint32_t fb[PB][2][4];
#pragma unroll
      for (int p = 0; p < PB; ++p)
#pragma unroll
        for (int n = 0; n < 2; ++n) OB::frag_b(Bs + p * OB::PART, wn + 16 * n, ks, lane, fb[p][n]);
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int pa = PA - 1; pa >= 0; --pa) { // small parts first
          uint32_t fa[4];
          OA::frag_a(As + pa * OA::PART, wm + 16 * m, ks, lane, fa);
#pragma unroll
          for (int pb = PB - 1; pb >= 0; --pb)
            if (pa + pb <= 2)
#pragma unroll
              for (int n = 0; n < 4; ++n)
                mma_bf16(c[m][n], fa, fb[pb][n >> 1][2 * (n & 1)], fb[pb][n >> 1][2 * (n & 1) + 1]);
        }
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[m][n][i] += c[m][n][i];
    }
    buf ^= 1;
    kt = nxt;
  }
  const bool atomic = g.splits > 1;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int hr = 0; hr < 2; ++hr) {
      const int m = m0 + wm + 16 * i + 8 * hr + (lane >> 2);
      if (m >= op.M) continue;
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int col = n0 + wn + 8 * n + 2 * (lane & 3) + e;
          if (col >= op.N) continue;
          float* dst = C + (int64_t)m * op.ldc + col;
          const float v = g.alpha * acc[i][n][2 * hr + e];
          if (atomic) atomicAdd(dst, v);
          else *dst = g.accumulate ? *dst + v : v;
        }
    }
}

template <typename TA, typename TB, bool AK, bool BK, bool CHAIN = false>
cudaError_t run_gemm(const GemmArgs& g, cudaStream_t s) {
  int M = 0, N = 0;
  for (int i = 0; i < g.ops; ++i) {
    M = std::max(M, g.op[i].M);
    N = std::max(N, g.op[i].N);
  }
  if (M <= 0 || N <= 0 || g.batch <= 0) return cudaSuccess;
  using OA = Operand<TA, AK>;
  using OB = Operand<TB, BK>;
  auto kern = bgemm_kernel<TA, TB, AK, BK, CHAIN>;
  constexpr int sm = 2 * (OA::PARTS * OA::PART + OB::PARTS * OB::PART) * 2;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  if (e != cudaSuccess) return e;
  dim3 grid((N + kBN - 1) / kBN, (M + kBM - 1) / kBM,
                  (CHAIN ? 1 : g.ops) * g.batch * g.splits);
  launch_pdl(kern, grid, dim3(kGemmThreads), (size_t)sm, s, g);
  return cudaGetLastError();
}

// Split K so that small outputs with long K still cover the SMs.
int choose_splits(int M, int N, int K, int batch) {
  const int64_t tiles = (int64_t)((M + kBM - 1) / kBM) * ((N + kBN - 1) / kBN) * batch;
  const int64_t want = 2LL * num_sms();
  if (tiles >= want) return 1;
  int s = (int)((want + tiles - 1) / tiles);
  const int maxs = max(1, K / (4 * kBK));      // keep at least 4 K tiles per split
  return max(1, min(s, min(maxs, 64)));
}

GemmArgs gemm_args(float alpha, int batch = 1, int64_t sa = 0, int64_t sb = 0, int64_t sc = 0) {
  GemmArgs g = {};
  g.sa = sa; g.sb = sb; g.sc = sc;
  g.batch = batch; g.splits = 1;
  g.alpha = alpha;
  return g;
}
void add_op(GemmArgs& g, const void* a, int64_t lda, const void* b, int64_t ldb, float* c,
            int64_t ldc, int M, int N, int K) {
  g.op[g.ops++] = GemmOp{a, b, c, M, N, K, lda, ldb, ldc};
}

// The fp32 outputs that splits add to, zeroed in one launch.
struct ZeroArgs {
  float* dst[12];
  int64_t n[12];
};
__global__ void __launch_bounds__(256) bwd_zero_kernel(const __grid_constant__ ZeroArgs a) {
  pdl_wait();
  pdl_trigger();
  float* dst = a.dst[blockIdx.y];
  const int64_t n = a.n[blockIdx.y];
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    dst[i] = 0.f;
}

// ---------------------------------------------------------------------------
// The reconstruction K_hat, V_hat [pairs][T][D] of pairs p0 .. p0 + npairs - 1
// (pair p = b Hkv + h) in fp32: one thread per 8 channels of a token.
// ---------------------------------------------------------------------------
__global__ void bwd_reconstruct_kernel(Geom g, int T, int p0, int npairs, float* kh, float* vh) {
  pdl_wait();
  const int c8 = g.D / 8;
  const int64_t n = (int64_t)npairs * T * c8;
  const int tq = g.fmt == KVQ_FMT_KIVI ? kivi_tq(T, g.R, g.G) : 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(i % c8);
    const int t = (int)((i / c8) % T);
    const int pp = (int)(i / ((int64_t)c8 * T));
    const int b = (p0 + pp) / g.H, h = (p0 + pp) % g.H;
    float* dst[2] = {kh + ((int64_t)pp * T + t) * g.D + 8 * c,
                     vh + ((int64_t)pp * T + t) * g.D + 8 * c};
    const bool raw = g.fmt == KVQ_FMT_FLOAT || (g.fmt == KVQ_FMT_KIVI && t >= tq);
    for (int which = 0; which < 2; ++which) {
      float v[8];
      if (raw && g.act == KVQ_F32) {
        const int slot = g.fmt == KVQ_FMT_KIVI ? t % g.ring : t;
        const float* src = plane_ptr<float>(g, which ? KVQ_PLANE_V_FULL : KVQ_PLANE_K_FULL, b, h,
                                            slot, 8 * c);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = src[e];
      } else {
        deq8(g, which, b, h, t, c, T, tq, v);
      }
#pragma unroll
      for (int e = 0; e < 8; e += 4)
        *reinterpret_cast<float4*>(dst[which] + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
    }
  }
}

// ---------------------------------------------------------------------------
// Per stacked query row: P = causal softmax(scale S) over S, and
// dS = P o (dP - sum_n P dP) scale over dP; masked entries become 0 as far as
// the products read them (the 64-row tile's last visible key, rounded up to a
// 64-key tile).  A warp per row: one pass for the running maximum, sum and
// sum of P dP, one that rewrites the row, 16 bytes a lane where the row length allows.
// Bound by HBM: S and dP are read twice (once from L2) and written once, the
// visible half only: 32000 rows of 1000 keys in 62 us (137 us with a CTA per row).
// Where T is no multiple of 4, rows are padded to one if the workspace has room for
// it and else taken element by element, here and in the products, with the same
// results: 1001 tokens (32 / 8 heads of 128, whole backward) 858 and 888 us.
// ---------------------------------------------------------------------------
constexpr int kRowWarps = 8;

// VEC: rows start on 16-byte boundaries (ld is a multiple of 4).
template <bool VEC>
__device__ __forceinline__ void row_load(const float* p, int left, float (&v)[4]) {
  if (VEC) {
    const float4 u = *reinterpret_cast<const float4*>(p);
    v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = i < left ? p[i] : 0.f;
  }
}
template <bool VEC>
__device__ __forceinline__ void row_store(float* p, int left, const float (&v)[4]) {
  if (VEC) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < left) p[i] = v[i];
  }
}

template <bool VEC>
__global__ void __launch_bounds__(kRowWarps * 32)
bwd_softmax_ds_kernel(float* S, float* dP, int M, int T, int ld, int L, float scale) {
  pdl_wait();
  pdl_trigger();
  const int m = blockIdx.x * kRowWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (m >= M) return;
  const int64_t row = ((int64_t)blockIdx.y * M + m) * ld;
  float* sp = S + row;
  float* dp = dP + row;
  const int nvis = T - L + m % L + 1;        // keys 0 .. T - L + l are visible
  const int tile = m / kBM * kBM;
  const int nend = min(T, (max_visible(tile, min(tile + kBM, M), L, T) / kBN + 1) * kBN);
  float mx = -INFINITY, sum = 0.f, dot = 0.f;
#pragma unroll 4
  for (int n = 4 * lane; n < nvis; n += 128) {
    float s[4], d[4];
    row_load<VEC>(sp + n, T - n, s);
    row_load<VEC>(dp + n, T - n, d);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (n + i >= nvis) s[i] = -INFINITY;
    const float top = fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3]));
    if (top > mx) {
      const float f = expf(scale * (mx - top));
      sum *= f;
      dot *= f;
      mx = top;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (n + i < nvis) {
        // (no finite score so far: an infinite one has weight 0, and -inf - -inf is NaN)
        const float e = s[i] == -INFINITY ? 0.f : expf(scale * (s[i] - mx));
        sum += e;
        dot = fmaf(e, d[i], dot);
      }
  }
  float top = mx;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
  const float f = mx == -INFINITY ? 0.f : expf(scale * (mx - top));
  sum *= f;
  dot *= f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    dot += __shfl_xor_sync(0xffffffffu, dot, o);
  }
  const float inv = 1.f / sum;
  const float delta = dot * inv;             // sum_n P dP
#pragma unroll 4
  for (int n = 4 * lane; n < nend; n += 128) {
    float s[4], d[4], p[4], ds[4];
    row_load<VEC>(sp + n, T - n, s);
    row_load<VEC>(dp + n, T - n, d);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      p[i] = ds[i] = 0.f;
      if (n + i < nvis) {
        p[i] = expf(scale * (s[i] - top)) * inv;
        ds[i] = p[i] * (d[i] - delta) * scale;
      }
    }
    row_store<VEC>(sp + n, T - n, p);
    row_store<VEC>(dp + n, T - n, ds);
  }
}

// ---------------------------------------------------------------------------
// Adapter backward: G [B L][(Hq + 2 Hkv) D], the gradient of the projection
// before RoPE (columns in w_qkv's row order).  d_k and d_v hold kv_rows
// tokens per (sequence, head), of which the last L are the tokens of x.
// ---------------------------------------------------------------------------
struct GatherArgs {
  const float* dq;
  const float* dk;
  const float* dv;
  float* G;
  int B, L, Hq, Hkv, D, kv_rows, pos0;
  float theta_hi[128], theta_lo[128];
};

// A thread has channels c, c + D/2 of one token for every head: the angle is
// formed once for all of them (with one sine and cosine per head, 1000 tokens x 48 heads of 128 took 44 us, now 15).
__global__ void __launch_bounds__(256) lora_gather_kernel(GatherArgs a) {
  pdl_wait();
  pdl_trigger();
  const int half = a.D / 2;
  const int heads = a.Hq + 2 * a.Hkv;
  const int64_t ntot = (int64_t)heads * a.D;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)a.B * a.L * half) return;
  const int c = (int)(i % half);
  const int64_t bl = i / half;
  const int b = (int)(bl / a.L), l = (int)(bl % a.L);
  float cs = 1.f, sn = 0.f;
  const bool rotate = a.theta_hi[0] != 0.f;
  if (rotate) pdec::rope_cos_sin(a.pos0 + l, a.theta_hi[c], a.theta_lo[c], &cs, &sn);
  const int64_t kv = ((int64_t)b * a.Hkv * a.kv_rows + (a.kv_rows - a.L + l)) * a.D;
  float* dst = a.G + bl * ntot;
  // heads blockIdx.y, blockIdx.y + gridDim.y, ...
#pragma unroll 4
  for (int hh = blockIdx.y; hh < heads; hh += gridDim.y) {
    const bool isv = hh >= a.Hq + a.Hkv;
    const float* src = hh < a.Hq ? a.dq + (((int64_t)b * a.Hq + hh) * a.L + l) * a.D
                                 : (isv ? a.dv : a.dk) + kv + (int64_t)((hh - a.Hq) % a.Hkv) * a.kv_rows * a.D;
    float g1 = src[c], g2 = src[c + half];
    if (rotate && !isv) {                     // the rotation transposed: angle -pos theta
      const float r1 = fmaf(g1, cs, g2 * sn);
      const float r2 = fmaf(g2, cs, -g1 * sn);
      g1 = r1;
      g2 = r2;
    }
    dst[(int64_t)hh * a.D + c] = g1;
    dst[(int64_t)hh * a.D + c + half] = g2;
  }
}

// Rows of G [rows][n] fp32, in place, as [rows][2n] bf16: the high parts
// (g rounded to bf16) then the bf16 of the remainders, so that the two halves
// carry about 16 significant bits of g for a bf16 tensor-core product.  One
// CTA per row at a time: the row goes through shared memory first.
__global__ void __launch_bounds__(256) bwd_split_rows_kernel(float* G, int rows, int n) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ float rowbuf[];
  for (int r = blockIdx.x; r < rows; r += gridDim.x) {
    float* g = G + (int64_t)r * n;
    for (int j = threadIdx.x; j < n; j += blockDim.x) rowbuf[j] = g[j];
    __syncthreads();
    __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(g);
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
      const float v = rowbuf[j];
      const __nv_bfloat16 hi = __float2bfloat16_rn(v);
      o[j] = hi;
      o[n + j] = __float2bfloat16_rn(v - __bfloat162float(hi));
    }
    __syncthreads();
  }
}

// Wt [d][n] = W [n][d] (bf16), 64 x 64 tiles through shared memory: 16-byte
// rows in, eight elements of a column gathered into each 16-byte store (n and d
// are multiples of 64).  6144 x 4096: 54 -> 17 us.
__global__ void __launch_bounds__(256) bwd_transpose_kernel(const __nv_bfloat16* __restrict__ W,
                                                            __nv_bfloat16* __restrict__ Wt, int n,
                                                            int d, int vec) {
  pdl_wait();
  pdl_trigger();
  __shared__ uint32_t tile[64][33];                         // 33 words: rows 8 apart in other banks
  const int n0 = blockIdx.y * 64, d0 = blockIdx.x * 64;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = (threadIdx.x >> 3) + 32 * i, c = threadIdx.x & 7;
    const __nv_bfloat16* src = W + (int64_t)(n0 + r) * d + d0 + 8 * c;
    __align__(16) __nv_bfloat16 e[8];
    if (vec) {
      *reinterpret_cast<uint4*>(e) = *reinterpret_cast<const uint4*>(src);
    } else {                                                // W off a 16-byte boundary
#pragma unroll
      for (int k = 0; k < 8; ++k) e[k] = src[k];
    }
    const uint4 u = *reinterpret_cast<const uint4*>(e);
    tile[r][4 * c] = u.x; tile[r][4 * c + 1] = u.y; tile[r][4 * c + 2] = u.z; tile[r][4 * c + 3] = u.w;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = (threadIdx.x >> 3) + 32 * i, c = threadIdx.x & 7;   // row of Wt, 8 columns from 8 c
    const uint32_t sel = r & 1 ? 0x7632 : 0x5410;
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      w[k] = __byte_perm(tile[8 * c + 2 * k][r >> 1], tile[8 * c + 2 * k + 1][r >> 1], sel);
    *reinterpret_cast<uint4*>(Wt + (int64_t)(d0 + r) * n + n0 + 8 * c) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

int grid_for(int64_t n, int threads) {
  const int64_t blocks = (n + threads - 1) / threads;
  return (int)std::min<int64_t>(blocks, (int64_t)num_sms() * 16);
}

}  // namespace

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
namespace {

// run_gemm with the activation-typed operand(s) chosen by `act`.
template <bool AK, bool BK, bool CHAIN = false>
cudaError_t gemm_act_b(const GemmArgs& g, int act, cudaStream_t s) {   // B in act dtype
  return act == KVQ_BF16 ? run_gemm<float, __nv_bfloat16, AK, BK, CHAIN>(g, s)
                         : run_gemm<float, float, AK, BK, CHAIN>(g, s);
}
template <bool AK, bool BK>
cudaError_t gemm_act_a(const GemmArgs& g, int act, cudaStream_t s) {   // A in act dtype
  return act == KVQ_BF16 ? run_gemm<__nv_bfloat16, float, AK, BK>(g, s)
                         : run_gemm<float, float, AK, BK>(g, s);
}
template <bool AK, bool BK>
cudaError_t gemm_act_ab(const GemmArgs& g, int act, cudaStream_t s) {  // both in act dtype
  return act == KVQ_BF16 ? run_gemm<__nv_bfloat16, __nv_bfloat16, AK, BK>(g, s)
                         : run_gemm<float, float, AK, BK>(g, s);
}

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

// (rows of S and dP of ld floats)
static size_t pair_bytes(const Geom& g, int T, int L, int ld) {
  const size_t gl = (size_t)(g.Hq / g.H) * L;
  return a256((2 * (size_t)T * g.D + 2 * gl * ld) * sizeof(float));
}
size_t attend_backward_pair_bytes(const Geom& g, int T, int L) { return pair_bytes(g, T, L, T); }

cudaError_t launch_attend_backward(const Geom& g, int T, const void* q, const void* d_out,
                                   int L, float scale, float* dq, float* dk, float* dv,
                                   void* ws, size_t ws_bytes, cudaStream_t s) {
  const int pairs = g.B * g.H, grp = g.Hq / g.H, D = g.D;
  const int M = grp * L;
  const int act = g.act, ld4 = (T + 3) & ~3;
  const size_t esz = act == KVQ_BF16 ? 2 : 4;
  // (two products of every pair share a launch: grid.z is at most 65,535)
  const int chunk = (int)std::min<size_t>(std::min(pairs, 65535 / 2),
                                          ws_bytes / pair_bytes(g, T, L, T));
  const int ld = chunk * pair_bytes(g, T, L, ld4) <= ws_bytes ? ld4 : T;
  cudaError_t e = cudaSuccess;
  for (int p0 = 0; p0 < pairs && e == cudaSuccess; p0 += chunk) {
    const int np = std::min(chunk, pairs - p0);
    float* kh = static_cast<float*>(ws);
    float* vh = kh + (size_t)np * T * D;
    float* S = vh + (size_t)np * T * D;
    float* dP = S + (size_t)np * M * ld;
    const char* qp = static_cast<const char*>(q) + (size_t)p0 * M * D * esz;
    const char* op = static_cast<const char*>(d_out) + (size_t)p0 * M * D * esz;
    launch_pdl(bwd_reconstruct_kernel, dim3(grid_for((int64_t)np * T * D / 8, 256)), dim3(256),
               0, s, g, T, p0, np, kh, vh);
    e = cudaGetLastError();
    // S = Q K^T and dP = dO V^T (tiles above the causal edge skipped)
    GemmArgs ga = gemm_args(1.f, np, (int64_t)M * D, (int64_t)T * D, (int64_t)M * ld);
    add_op(ga, qp, D, kh, D, S, ld, M, T, D);
    add_op(ga, op, D, vh, D, dP, ld, M, T, D);
    ga.mask = kMaskRowsQueriesColsKeys; ga.L = L; ga.T = T;
    if (e == cudaSuccess) e = gemm_act_a<true, true>(ga, act, s);
    if (e == cudaSuccess) {
      launch_pdl(ld % 4 == 0 ? bwd_softmax_ds_kernel<true> : bwd_softmax_ds_kernel<false>,
                 dim3((M + kRowWarps - 1) / kRowWarps, np), dim3(kRowWarps * 32), 0, s, S, dP, M, T,
                 ld, L, scale);
      e = cudaGetLastError();
    }
    // dQ = dS K
    GemmArgs gq = gemm_args(1.f, np, (int64_t)M * ld, (int64_t)T * D, (int64_t)M * D);
    add_op(gq, dP, ld, kh, D, dq + (size_t)p0 * M * D, D, M, D, T);
    gq.mask = kMaskRowsQueriesKKeys; gq.L = L; gq.T = T;
    if (e == cudaSuccess) e = run_gemm<float, float, true, false>(gq, s);
    // dK = dS^T Q and dV = P^T dO
    GemmArgs gk = gemm_args(1.f, np, (int64_t)M * ld, (int64_t)M * D, (int64_t)T * D);
    add_op(gk, dP, ld, qp, D, dk + (size_t)p0 * T * D, D, T, D, M);
    add_op(gk, S, ld, op, D, dv + (size_t)p0 * T * D, D, T, D, M);
    gk.mask = kMaskRowsKeysKQueries; gk.L = L; gk.T = T;
    if (e == cudaSuccess) e = gemm_act_b<false, false>(gk, act, s);
  }
  return e;
}

size_t lora_backward_bytes(int B, int L, int d_in, int Hq, int Hkv, int D, const int r[3]) {
  const size_t BL = (size_t)B * L;
  size_t n = a256(BL * (Hq + 2 * Hkv) * D * sizeof(float));
  for (int p = 0; p < 3; ++p) n += 2 * a256(BL * r[p] * sizeof(float));
  n += a256((size_t)d_in * (Hq + 2 * Hkv) * D * 2);   // W^T in bf16 for the d_x product
  return n;
}

// d_x on tcgen05 needs bf16 activations and whole 64-element K slices and
// 128-column output tiles.
static bool dx_on_tc(int act, int d_in, int ntot) {
  return act == KVQ_BF16 && d_in % 128 == 0 && ntot % 64 == 0;
}

cudaError_t launch_lora_backward(const void* x, int B, int L, int d_in, const void* w,
                                 const void* const a[3], const void* const bm[3],
                                 const int r[3], float alpha_over_r, int Hq, int Hkv, int D,
                                 int pos0, float rope_base, int act, const float* dq,
                                 const float* dk, const float* dv, int kv_rows,
                                 float* const da[3], float* const db[3], float* dx, void* ws,
                                 cudaStream_t s) {
  const int BL = B * L;
  const int ntot = (Hq + 2 * Hkv) * D;
  const int nout[3] = {Hq * D, Hkv * D, Hkv * D};
  const int off[3] = {0, Hq * D, (Hq + Hkv) * D};
  char* wp = static_cast<char*>(ws);
  float* G = reinterpret_cast<float*>(wp);
  wp += a256((size_t)BL * ntot * sizeof(float));
  float* U[3];
  float* V[3];
  for (int p = 0; p < 3; ++p) {
    U[p] = reinterpret_cast<float*>(wp);
    wp += a256((size_t)BL * r[p] * sizeof(float));
    V[p] = reinterpret_cast<float*>(wp);
    wp += a256((size_t)BL * r[p] * sizeof(float));
  }
  __nv_bfloat16* Wt = reinterpret_cast<__nv_bfloat16*>(wp);   // [d_in][ntot]
  GatherArgs ga;
  ga.dq = dq; ga.dk = dk; ga.dv = dv; ga.G = G;
  ga.B = B; ga.L = L; ga.Hq = Hq; ga.Hkv = Hkv; ga.D = D; ga.kv_rows = kv_rows; ga.pos0 = pos0;
  rope_theta_table(rope_base, D, ga.theta_hi, ga.theta_lo);
  const int tblocks = (int)(((int64_t)BL * D / 2 + 255) / 256);
  const int hblocks = std::max(1, std::min(Hq + 2 * Hkv, 8 * num_sms() / tblocks));   // cover the SMs
  launch_pdl(lora_gather_kernel, dim3(tblocks, hblocks), dim3(256), 0, s, ga);
  cudaError_t e = cudaGetLastError();
  // per projection: U_p = x A_p^T and V_p = g_p B_p [BL][r] (narrow outputs over
  // long K), dB_p = (alpha/r) g_p^T U_p [n_p][r], dA_p = (alpha/r) V_p^T x [r][d_in]
  // (over the BL rows): split over K, added atomically into zeroed outputs
  GemmArgs gu = gemm_args(1.f), gv = gemm_args(1.f), gb = gemm_args(alpha_over_r),
           gA = gemm_args(alpha_over_r), gl = gemm_args(alpha_over_r);
  int rmax = 0, nmax = 0;
  for (int p = 0; p < 3; ++p) {
    if (r[p] == 0) continue;
    add_op(gu, x, d_in, a[p], d_in, U[p], r[p], BL, r[p], d_in);
    add_op(gv, G + off[p], ntot, bm[p], r[p], V[p], r[p], BL, r[p], nout[p]);
    add_op(gb, G + off[p], ntot, U[p], r[p], db[p], r[p], nout[p], r[p], BL);
    add_op(gA, V[p], r[p], x, d_in, da[p], d_in, r[p], d_in, BL);
    add_op(gl, V[p], r[p], a[p], d_in, dx, d_in, BL, d_in, r[p]);
    rmax = std::max(rmax, r[p]);
    nmax = std::max(nmax, nout[p]);
  }
  if (gu.ops > 0 && e == cudaSuccess) {
    gu.splits = choose_splits(BL, rmax, d_in, gu.ops);
    gv.splits = choose_splits(BL, rmax, nmax, gv.ops);
    gb.splits = choose_splits(nmax, rmax, BL, gb.ops);
    gA.splits = choose_splits(rmax, d_in, BL, gA.ops);
    ZeroArgs z = {};
    int nz = 0;
    for (const GemmArgs* gg : {&gu, &gv, &gb, &gA})
      for (int i = 0; i < gg->ops && gg->splits > 1; ++i) {
        z.dst[nz] = gg->op[i].c;
        z.n[nz++] = (int64_t)gg->op[i].M * gg->op[i].N;
      }
    if (nz > 0) {
      launch_pdl(bwd_zero_kernel, dim3(32, nz), dim3(256), 0, s, z);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = gemm_act_ab<true, true>(gu, act, s);
    if (e == cudaSuccess) e = gemm_act_b<true, false>(gv, act, s);
    if (e == cudaSuccess) e = run_gemm<float, float, false, false>(gb, s);
    if (e == cudaSuccess) e = gemm_act_b<false, false>(gA, act, s);
  }
  if (dx && e == cudaSuccess) {
    // dx = g W + sum_p (alpha/r) V_p A_p
    // (the tensor-core product stores 16 bytes at a time)
    if (dx_on_tc(act, d_in, ntot) && (reinterpret_cast<uintptr_t>(dx) & 15) == 0) {
      // g W on tcgen05: g split into bf16 high and low parts in place (G is
      // not read again), [g_hi | g_lo] times [W^T | W^T] along K
      int* err = device_error_word();
      if (!err) return cudaErrorInvalidDevice;
      launch_pdl(bwd_transpose_kernel, dim3(d_in / 64, ntot / 64), dim3(256), 0, s,
                 reinterpret_cast<const __nv_bfloat16*>(w), Wt, ntot, d_in,
                 (reinterpret_cast<uintptr_t>(w) & 15) == 0 ? 1 : 0);
      e = cudaGetLastError();
      const size_t sm = (size_t)ntot * sizeof(float);
      if (e == cudaSuccess && sm > 48 * 1024)
        e = cudaFuncSetAttribute(bwd_split_rows_kernel,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (e == cudaSuccess) {
        launch_pdl(bwd_split_rows_kernel, dim3(std::min(BL, num_sms() * 8)), dim3(256), sm, s, G,
                   BL, ntot);
        e = cudaGetLastError();
      }
      if (e == cudaSuccess) e = launch_gemm_tc_bf16(G, BL, 2 * ntot, Wt, d_in, ntot, dx, err, s);
    } else {
      GemmArgs gx = gemm_args(1.f);
      add_op(gx, G, ntot, w, d_in, dx, d_in, BL, d_in, ntot);
      e = gemm_act_b<true, false>(gx, act, s);
    }
    // the adapters' part, sum_p V_p A_p, in one pass over dx
    if (gl.ops > 0 && e == cudaSuccess) {
      gl.accumulate = 1;
      e = gemm_act_b<true, false, true>(gl, act, s);
    }
  }
  return e;
}

}  // namespace kvq
