// LoRA-adapted Q/K/V projection (Section 3, Eq. 1 and Eq. lora) with rotary
// positions, written head-major.  The adapter stays an explicit rank-r
// branch (Section 3.4): y = x W^T + (alpha/r) (x A^T) B^T.
#include <math.h>

#include "proj_decode.cuh"

namespace kvq {
// The weight-streaming decode projection (proj_stream.cu); cudaErrorNotSupported
// when the shape is outside its range (M > 16, d_in > 4096, rank > 64).
cudaError_t launch_project_decode_stream(const pdec::ProjArgs& p, int* err, cudaStream_t s);
}  // namespace kvq

namespace kvq {
namespace {
using namespace pdec;

constexpr int kMT = 32;     // rows per CTA
constexpr int kNT = 64;     // output columns per CTA: 32 RoPE pairs of one head
constexpr int kKC = 32;     // k chunk
constexpr int kThreads = 128;

// Elements k .. k + 3 of a row (zeros from K on).
template <typename T>
__device__ __forceinline__ float4 load4(const T* row, int k, int K, bool vec);
template <>
__device__ __forceinline__ float4 load4<float>(const float* row, int k, int K, bool vec) {
  if (vec) return k < K ? *reinterpret_cast<const float4*>(row + k) : make_float4(0.f, 0.f, 0.f, 0.f);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (k < K) v.x = row[k];
  if (k + 1 < K) v.y = row[k + 1];
  if (k + 2 < K) v.z = row[k + 2];
  if (k + 3 < K) v.w = row[k + 3];
  return v;
}
template <>
__device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* row, int k, int K, bool) {
  if (k >= K) return make_float4(0.f, 0.f, 0.f, 0.f);       // K is a multiple of 64
  const uint2 u = *reinterpret_cast<const uint2*>(row + k);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

// More than 16 rows, fp32 (and the bf16 head shapes the tensor-core kernel does
// not tile): one CTA = kMT rows of x times 32 channel pairs (c, c + D/2) of one
// head, a thread 4 rows x 2 pairs in registers.  The rank-r product x A_p^T rides
// along as up to 64 further columns, so x is read once per CTA; every output
// is one fp32 chain over k in order, then over the ranks.
// What bounds it at these sizes (512 rows x 768 outputs x 256 inputs: 0.2
// GFLOP) is the chain of k chunks: small tiles keep 192 CTAs in flight and the
// next chunk's loads go out before the current one is multiplied: 129 us with
// one shared-memory read per multiplication, 29 us so.
template <typename T>
__global__ void __launch_bounds__(kThreads) project_tile_kernel(ProjArgs p) {
  pdl_wait();
  pdl_trigger();
  __shared__ __align__(16) float Xs[2][kKC][kMT + 4];
  __shared__ __align__(16) float Ws[2][kKC][kNT + 4];
  __shared__ __align__(16) float As[2][kKC][64 + 4];        // then (alpha/r) x A^T [kMT][68]
  const int D = p.D, M = p.B * p.L, K = p.d_in, half = D / 2;
  const int tiles = D / kNT;                 // column tiles per head
  const int hh = blockIdx.y / tiles;         // stacked head index over q, k, v
  const int c0 = blockIdx.y % tiles * (kNT / 2);
  const int proj = hh < p.Hq ? 0 : hh < p.Hq + p.Hkv ? 1 : 2;
  const int head = proj == 0 ? hh : proj == 1 ? hh - p.Hq : hh - p.Hq - p.Hkv;
  const int r = p.r[proj], ne = (r + 15) / 16;
  const int m0 = blockIdx.x * kMT;
  const bool vec = sizeof(T) == 2 || K % 4 == 0;
  const T* x = reinterpret_cast<const T*>(p.x);
  const T* w = reinterpret_cast<const T*>(p.w);
  const T* am = reinterpret_cast<const T*>(p.a[proj]);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  // operand rows of this thread: x row tid % 32, W rows tid % 64, A rows tid % 64,
  // at k chunks of 4 tid / 32 (x) or tid / 64 + 2 i (W, A)
  const int xr = tid & 31, xk = (tid >> 5) * 4;
  const int wr = tid & 63, wk = (tid >> 6) * 4;
  const bool xin = m0 + xr < M, ain = wr < r;
  const T* xrow = x + (int64_t)(xin ? m0 + xr : 0) * K;
  const T* wrow = w + ((int64_t)hh * D + (wr < 32 ? c0 + wr : half + c0 + wr - 32)) * K;
  const T* arow = am + (int64_t)(ain ? wr : 0) * K;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 xv[2], wv[4], av[4];
  auto load = [&](int k0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) xv[i] = xin ? load4<T>(xrow, k0 + xk + 16 * i, K, vec) : zero;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      wv[i] = load4<T>(wrow, k0 + wk + 8 * i, K, vec);
      av[i] = ain ? load4<T>(arow, k0 + wk + 8 * i, K, vec) : zero;
    }
  };
  auto put = [](float (*s)[kNT + 4], int k, int row, const float4& v) {
    s[k][row] = v.x;
    s[k + 1][row] = v.y;
    s[k + 2][row] = v.z;
    s[k + 3][row] = v.w;
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int k = xk + 16 * i;
      Xs[buf][k][xr] = xv[i].x;
      Xs[buf][k + 1][xr] = xv[i].y;
      Xs[buf][k + 2][xr] = xv[i].z;
      Xs[buf][k + 3][xr] = xv[i].w;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      put(Ws[buf], wk + 8 * i, wr, wv[i]);
      if (ne) put(As[buf], wk + 8 * i, wr, av[i]);
    }
  };
  float acc[4][4] = {}, uacc[4][4] = {};     // [row][2 tx, 2 tx + 1, their partners], [row][16 e + tx]
  const int chunks = (K + kKC - 1) / kKC;
  load(0);
  for (int c = 0; c < chunks; ++c) {
    const int buf = c & 1;
    store(buf);
    __syncthreads();
    if (c + 1 < chunks) load((c + 1) * kKC);
#pragma unroll 8
    for (int k = 0; k < kKC; ++k) {
      const float4 xq = *reinterpret_cast<const float4*>(&Xs[buf][k][4 * ty]);
      const float2 w0 = *reinterpret_cast<const float2*>(&Ws[buf][k][2 * tx]);
      const float2 w1 = *reinterpret_cast<const float2*>(&Ws[buf][k][32 + 2 * tx]);
      const float xm[4] = {xq.x, xq.y, xq.z, xq.w}, wn[4] = {w0.x, w0.y, w1.x, w1.y};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xm[i], wn[j], acc[i][j]);
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (e < ne) {
          const float ae = As[buf][k][16 * e + tx];
#pragma unroll
          for (int i = 0; i < 4; ++i) uacc[i][e] = fmaf(xm[i], ae, uacc[i][e]);
        }
    }
    // (the other buffer is free: every thread passed this chunk's barrier
    // after it had finished the chunk before)
  }
  // + (alpha/r) (x A^T) B^T
  if (r > 0) {
    float (*U)[68] = reinterpret_cast<float (*)[68]>(&As[0][0][0]);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) U[4 * ty + i][16 * e + tx] = uacc[i][e] * p.alpha_over_r;
    __syncthreads();
    const T* bm = reinterpret_cast<const T*>(p.bm[proj]);
    const int ch[4] = {c0 + 2 * tx, c0 + 2 * tx + 1, half + c0 + 2 * tx, half + c0 + 2 * tx + 1};
    for (int j = 0; j < r; ++j) {
      float bv[4];
#pragma unroll
      for (int n = 0; n < 4; ++n) bv[n] = (float)bm[((int64_t)head * D + ch[n]) * r + j];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float u = U[4 * ty + i][j];
#pragma unroll
        for (int n = 0; n < 4; ++n) acc[i][n] = fmaf(u, bv[n], acc[i][n]);
      }
    }
  }
  // RoPE (rotate-half) on q and k, head-major store
  const bool rope = proj < 2 && p.rope_base > 0.f;
  const int H = proj == 0 ? p.Hq : p.Hkv;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int gm = m0 + 4 * ty + i;
    if (gm >= M) continue;
    const int b = gm / p.L, l = gm % p.L;
    const int64_t o = (((int64_t)b * H + head) * p.L + l) * D + c0 + 2 * tx;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      float y1 = acc[i][j], y2 = acc[i][2 + j];
      if (rope) {
        float c, s;
        const int fi = c0 + 2 * tx + j;
        rope_cos_sin(p.pos0 + pos_of(p.pos_dev, p.pos_stride, b) + l, p.theta_hi[fi], p.theta_lo[fi],
                     &c, &s);
        const float r1 = y1 * c - y2 * s, r2 = y2 * c + y1 * s;
        y1 = r1;
        y2 = r2;
      }
      st_act(p.out[proj], o + j, y1, p.act);
      st_act(p.out[proj], o + half + j, y2, p.act);
    }
  }
}

// ---------------------------------------------------------------------------
// Few rows (M = B * L <= 16, the decode step): weight streaming.  Each warp
// owns one RoPE column pair (c, c + D/2) of one head and streams both weight
// rows with 16-byte loads; x (all M rows) sits in shared memory.  The
// rank-r branch: the CTA first forms (alpha/r) x A_p^T for its projection.
// ---------------------------------------------------------------------------
constexpr int kSkinnyWarps = 4;      // 3 CTAs per SM: one wave for up to 456 CTAs
constexpr int kSkinnyMaxM = 16;
constexpr int kSkinnyKIter = 8;      // 16-byte loads per row per lane in flight (2048 bf16)

template <typename T>
__device__ __forceinline__ void load8f(const T* p, float f[8]);
template <>
__device__ __forceinline__ void load8f<__nv_bfloat16>(const __nv_bfloat16* p, float f[8]) {
  uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float2 t = __bfloat1622float2(h[i]);
    f[2 * i] = t.x;
    f[2 * i + 1] = t.y;
  }
}
template <>
__device__ __forceinline__ void load8f<float>(const float* p, float f[8]) {
  float4 a = __ldg(reinterpret_cast<const float4*>(p));
  float4 b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}

// Raw 8-element vector of activation type T (kept packed until used).
template <typename T> struct Raw8;
template <> struct Raw8<__nv_bfloat16> {
  uint4 u;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) {
    u = __ldg(reinterpret_cast<const uint4*>(p));
  }
  __device__ __forceinline__ void to_float(float f[8]) const {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float2 t = __bfloat1622float2(h[i]);
      f[2 * i] = t.x;
      f[2 * i + 1] = t.y;
    }
  }
};
template <> struct Raw8<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p) {
    a = __ldg(reinterpret_cast<const float4*>(p));
    b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  }
  __device__ __forceinline__ void to_float(float f[8]) const {
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
  }
};

template <typename T, int MM, int KITER>
__global__ void __launch_bounds__(kSkinnyWarps * 32, 3) project_skinny_kernel(ProjArgs p) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ float xsm[];             // [M][d_in] fp32, then U [M][64]
  const int M = p.B * p.L, D = p.D, K = p.d_in;
  const int half = D / 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pairs_per_head = half;
  const int pair0 = blockIdx.x * kSkinnyWarps;      // CTA's first pair (stacked heads)
  const int hh = pair0 / pairs_per_head;           // all 8 pairs of a CTA share a head
  const int proj = hh < p.Hq ? 0 : hh < p.Hq + p.Hkv ? 1 : 2;
  const int head = proj == 0 ? hh : proj == 1 ? hh - p.Hq : hh - p.Hq - p.Hkv;
  const int r = p.r[proj];
  float* U = xsm + M * K;
  const T* x = reinterpret_cast<const T*>(p.x);
  const int c = (pair0 + warp) % pairs_per_head;    // channel within the first half
  const int n1 = hh * D + c, n2 = n1 + half;
  const T* W = reinterpret_cast<const T*>(p.w);
  const T* w1 = W + (int64_t)n1 * K;
  const T* w2 = W + (int64_t)n2 * K;
  // x -> shared memory (fp32): every thread issues all its loads, then stores
  {
    constexpr int XL = 8;                           // 16-byte loads per thread per round
    for (int base = threadIdx.x * 8; base < M * K; base += blockDim.x * 8 * XL) {
      Raw8<T> xv[XL];
#pragma unroll
      for (int u = 0; u < XL; ++u) {
        const int i = base + u * blockDim.x * 8;
        if (i < M * K) xv[u].load(x + i);
      }
#pragma unroll
      for (int u = 0; u < XL; ++u) {
        const int i = base + u * blockDim.x * 8;
        if (i < M * K) {
          float f[8];
          xv[u].to_float(f);
          *reinterpret_cast<float4*>(xsm + i) = make_float4(f[0], f[1], f[2], f[3]);
          *reinterpret_cast<float4*>(xsm + i + 4) = make_float4(f[4], f[5], f[6], f[7]);
        }
      }
    }
  }
  __syncthreads();
  // x A_p^T, one warp per rank: the row's 16-byte loads are all in flight
  // (passes of KITER x 256 channels), then M dot products reduced by shuffles.
  if (r > 0) {
    const T* A = reinterpret_cast<const T*>(p.a[proj]);
    for (int j = warp; j < r; j += kSkinnyWarps) {
      float acc[MM];
#pragma unroll
      for (int m = 0; m < MM; ++m) acc[m] = 0.f;
      for (int kp = 0; kp < K; kp += KITER * 256) {
        Raw8<T> av[KITER];
#pragma unroll
        for (int u = 0; u < KITER; ++u) {
          const int k = kp + lane * 8 + u * 256;
          if (k < K) av[u].load(A + (int64_t)j * K + k);
        }
#pragma unroll
        for (int u = 0; u < KITER; ++u) {
          const int k = kp + lane * 8 + u * 256;
          if (k < K) {
            float a[8];
            av[u].to_float(a);
#pragma unroll
            for (int m = 0; m < MM; ++m) {
              if (m < M) {
                const float4* xr4 = reinterpret_cast<const float4*>(xsm + m * K + k);
                const float4 xa = xr4[0], xb = xr4[1];
                acc[m] += a[0] * xa.x + a[1] * xa.y + a[2] * xa.z + a[3] * xa.w +
                          a[4] * xb.x + a[5] * xb.y + a[6] * xb.z + a[7] * xb.w;
              }
            }
          }
        }
      }
#pragma unroll
      for (int m = 0; m < MM; ++m) {
        float v = acc[m];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0 && m < M) U[m * 64 + j] = v;
      }
    }
  }
  // this warp's weight rows in passes of KITER x 256 channels: KITER 8-element
  // loads per row per lane in flight together (the bulk of the bytes)
  float acc1[MM], acc2[MM];
#pragma unroll
  for (int m = 0; m < MM; ++m) { acc1[m] = 0.f; acc2[m] = 0.f; }
  for (int kp = 0; kp < K; kp += KITER * 256) {
  Raw8<T> wa[KITER], wb[KITER];
#pragma unroll
  for (int u = 0; u < KITER; ++u) {
    const int k = kp + lane * 8 + u * 256;
    if (k < K) {
      wa[u].load(w1 + k);
      wb[u].load(w2 + k);
    }
  }
#pragma unroll
  for (int u = 0; u < KITER; ++u) {
    const int k = kp + lane * 8 + u * 256;
    if (k < K) {
      float a[8], bq[8];
      wa[u].to_float(a);
      wb[u].to_float(bq);
#pragma unroll
      for (int m = 0; m < MM; ++m) {
        if (m < M) {
          const float4* xr4 = reinterpret_cast<const float4*>(xsm + m * K + k);
          const float4 xa = xr4[0], xb = xr4[1];
          const float xr[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            acc1[m] += a[e] * xr[e];
            acc2[m] += bq[e] * xr[e];
          }
        }
      }
    }
  }
  }
#pragma unroll
  for (int m = 0; m < MM; ++m) {
    for (int o = 16; o > 0; o >>= 1) {
      acc1[m] += __shfl_xor_sync(0xffffffffu, acc1[m], o);
      acc2[m] += __shfl_xor_sync(0xffffffffu, acc2[m], o);
    }
  }
  __syncthreads();                                  // U complete
  // rank-r up projection, RoPE, head-major store: lane m handles row m
  if (lane < M) {
    float y1 = 0.f, y2 = 0.f;
#pragma unroll
    for (int m = 0; m < MM; ++m)
      if (m == lane) { y1 = acc1[m]; y2 = acc2[m]; }
    if (r > 0) {
      const T* Bm = reinterpret_cast<const T*>(p.bm[proj]);
      const T* b1 = Bm + ((int64_t)head * D + c) * r;
      const T* b2 = Bm + ((int64_t)head * D + c + half) * r;
      for (int j0 = 0; j0 < r; j0 += 8) {          // r is a multiple of 8
        float f1[8], f2[8];
        load8f<T>(b1 + j0, f1);
        load8f<T>(b2 + j0, f2);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float uu = U[lane * 64 + j0 + e] * p.alpha_over_r;
          y1 += uu * f1[e];
          y2 += uu * f2[e];
        }
      }
    }
    const int b = lane / p.L, l = lane % p.L;
    if (proj < 2 && p.rope_base > 0.f) {
      const int pos = p.pos0 + pos_of(p.pos_dev, p.pos_stride, b) + l;
      float cs, sn;
      rope_cos_sin(pos, p.theta_hi[c], p.theta_lo[c], &cs, &sn);
      const float o1 = y1 * cs - y2 * sn, o2 = y2 * cs + y1 * sn;
      y1 = o1;
      y2 = o2;
    }
    const int H = proj == 0 ? p.Hq : p.Hkv;
    const int64_t base = (((int64_t)b * H + head) * p.L + l) * D;
    st_act(p.out[proj], base + c, y1, p.act);
    st_act(p.out[proj], base + c + half, y2, p.act);
  }
}

template <int M16, int NT>
__global__ void __launch_bounds__(kDecWarps * 32) project_decode_mma_kernel(ProjArgs p) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char dsm[];
  proj_decode_tile<M16, NT>(p, blockIdx.x, dsm);
}

template <int M16, int NT>
cudaError_t launch_decode_mma_nt(const ProjArgs& p, cudaStream_t s) {
  const size_t sm = proj_decode_smem_bytes(M16, NT, p.d_in);
  auto kern = project_decode_mma_kernel<M16, NT>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  const int tiles = (p.Hq + 2 * p.Hkv) * (p.D / 16);
  launch_pdl(kern, dim3(tiles), dim3(kDecWarps * 32), sm, s, p);
  return cudaGetLastError();
}

cudaError_t launch_decode_mma(const ProjArgs& p, cudaStream_t s) {
  const int M = p.B * p.L;
  const int rmax = max(p.r[0], max(p.r[1], p.r[2]));
  const int nt = 2 + rmax / 8;
  if (M <= 8) {
    if (nt <= 4) return launch_decode_mma_nt<8, 4>(p, s);
    return launch_decode_mma_nt<8, kDecMaxNt>(p, s);
  }
  if (nt <= 4) return launch_decode_mma_nt<16, 4>(p, s);
  return launch_decode_mma_nt<16, kDecMaxNt>(p, s);
}

template <typename T>
cudaError_t launch_skinny(const ProjArgs& p, cudaStream_t s) {
  const int M = p.B * p.L;
  const int pairs = (p.Hq + 2 * p.Hkv) * p.D / 2;
  const size_t sm = ((size_t)M * p.d_in + (size_t)kSkinnyMaxM * 64) * sizeof(float);
  // fp32 weights take twice the registers: half the loads per pass
  constexpr int KI = sizeof(T) == 2 ? kSkinnyKIter : kSkinnyKIter / 2;
  auto kern = M <= 4 ? project_skinny_kernel<T, 4, KI>
            : M <= 8 ? project_skinny_kernel<T, 8, KI> : project_skinny_kernel<T, kSkinnyMaxM, KI>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  launch_pdl(kern, dim3(pairs / kSkinnyWarps), dim3(kSkinnyWarps * 32), sm, s, p);
  return cudaGetLastError();
}

}  // namespace

// RoPE frequencies base^(-2i/D) for i < D/2 in fp64, split into hi + lo
// floats (zeros elsewhere, or everywhere when base = 0).
void rope_theta_table(float rope_base, int D, float* hi, float* lo) {
  for (int i = 0; i < 128; ++i) {
    const double th = i < D / 2 && rope_base > 0.f ? pow((double)rope_base, -2.0 * i / D) : 0.0;
    hi[i] = (float)th;
    lo[i] = (float)(th - (double)hi[i]);
  }
}

cudaError_t launch_project(const void* x, int B, int L, int d_in, const void* w,
                           const void* const a[3], const void* const bm[3], const int r[3],
                           float alpha_over_r, int Hq, int Hkv, int D, int pos0,
                           const int* pos_dev, float rope_base, int act,
                           void* const out[3], int* err, cudaStream_t s, int pos_stride) {
  ProjArgs p;
  p.x = x; p.w = w;
  for (int i = 0; i < 3; ++i) { p.a[i] = a[i]; p.bm[i] = bm[i]; p.r[i] = r[i]; p.out[i] = out[i]; }
  p.B = B; p.L = L; p.d_in = d_in; p.Hq = Hq; p.Hkv = Hkv; p.D = D; p.pos0 = pos0; p.act = act;
  p.pos_dev = pos_dev;
  p.pos_stride = pos_stride;
  p.alpha_over_r = alpha_over_r; p.rope_base = rope_base;
  rope_theta_table(rope_base, D, p.theta_hi, p.theta_lo);
  const int M = B * L;
  if (act == KVQ_BF16 && M > kSkinnyMaxM) {
    cudaError_t e = launch_project_tc(x, B, L, d_in, w, a, bm, r, alpha_over_r, Hq, Hkv, D, pos0,
                                      pos_dev, rope_base, out, err, s, nullptr, pos_stride);
    if (e != cudaErrorNotSupported) return e;
    (void)cudaGetLastError();
  }
  if (act == KVQ_BF16 && M <= 16 && d_in % 64 == 0) {
    cudaError_t e = launch_project_decode_stream(p, err, s);
    if (e != cudaErrorNotSupported) return e;
    (void)cudaGetLastError();
  }
  if (act == KVQ_BF16 && M <= 16 && d_in % 32 == 0 && (size_t)16 * d_in * 2 <= 160 * 1024)
    return launch_decode_mma(p, s);
  if (M <= kSkinnyMaxM && (size_t)M * d_in * 4 <= 120 * 1024 && d_in % 64 == 0)
    return act == KVQ_BF16 ? launch_skinny<__nv_bfloat16>(p, s) : launch_skinny<float>(p, s);
  const dim3 grid((M + kMT - 1) / kMT, (Hq + 2 * Hkv) * (D / kNT));
  if (act == KVQ_BF16) launch_pdl(project_tile_kernel<__nv_bfloat16>, grid, dim3(kThreads), 0, s, p);
  else launch_pdl(project_tile_kernel<float>, grid, dim3(kThreads), 0, s, p);
  return cudaGetLastError();
}

}  // namespace kvq
