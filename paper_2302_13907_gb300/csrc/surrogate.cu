// Trace surrogate: a small MLP + transposed-convolution decoder trained and
// run with hand-written kernels.
//
//   h1 = gelu(x W1 + b1)                      6 -> H1
//   h2 = gelu(h1 W2 + b2)                     H1 -> H2
//   a0 = gelu(reshape(h2 W3 + b3, [L0, C0]))  channels last
//   a_{l+1} = gelu(convT(a_l; T_l, t_l))      kernel 4, stride 2, padding 1
//   y = a_5 Wf + bf                           1x1 convolution to 8 receivers
//
// Every contraction is a GEMM on the tensor cores (BF16 operands, FP32
// accumulation): dense layers directly; a transposed convolution as
// Z = a T (T viewed as [C_in][C_out*4]) followed by a col2im sum of the two
// taps landing on each output position; its backward as im2col + two GEMMs.
// Weights are kept as FP32 masters (Adam) with BF16 copies for the GEMMs;
// activations are BF16 at every GEMM input, FP32 elsewhere.
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "../../include/cwell.h"
#include "cwell_internal.cuh"

namespace cwell {

// ------------------------------------------------------------------ GEMM
// C[M x N] = op(A)[M x K] * op(B)[K x N], A and B BF16 row-major (op =
// transpose when TA / TB), C FP32 row-major.  64 x 64 tiles, K step 32, four
// warps of 32 x 32, mma.sync m16n8k16 (BF16 in, FP32 acc).
//
// The products here have a few MFLOP, so what bounds them is the latency of
// one block's walk along K.  Operand tiles are staged four deep with 16-byte
// cp.async in the layout of their source ([row][k] or [k][row]; ldmatrix,
// transposing where K is not the contiguous index, forms the fragments), so
// three K steps of loads are in flight behind the MMAs (64 x 512 x 256 in 6.7
// us, 32 x 512 x 4096 in 54 us; 43 and 573 us with 2-byte loads staged one K
// step at a time).  Every element is one
// chain of MMAs over ascending K, as in gemm_wgrad below: the training
// amplifies a changed order of the sum (Adam divides by the gradients' own
// size), so no product is cut along K.
constexpr int GBM = 64, GBN = 64, GBK = 32, GST = 4;
constexpr int GLD_K = GBK + 8, GLD_R = 64 + 8;  // row pitch of a [row][k] / [k][row] tile: ldmatrix rows in distinct banks
constexpr int GTILE = GBM * GLD_K;              // elements per staged tile (the larger of the two layouts)

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

template <bool TRANS>
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const __nv_bfloat16 *p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  if (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

// Stage a 64 (rows r0 .. of R) x 32 (k0 .. of kend) operand tile: KC = K is
// the contiguous index of the source (element (r, k) at src[r ld + k], tile
// [row][k]), otherwise element (r, k) at src[k ld + r], tile [k][row].  Eight
// contiguous elements at a time, zero outside; vec: rows of the source are
// 16-byte aligned (ld a multiple of 8, base aligned).
template <bool KC>
__device__ __forceinline__ void stage_tile(__nv_bfloat16 *tile, const __nv_bfloat16 *src, int ld, int r0, int R, int k0,
                                           int kend, bool vec) {
#pragma unroll
  for (int q = threadIdx.x; q < 256; q += 128) {
    const int r = KC ? q >> 2 : (q & 7) * 8, k = KC ? (q & 3) * 8 : q >> 3;
    const int gr = r0 + r, gk = k0 + k;
    const int left = KC ? kend - gk : R - gr;  // elements of the source row from here on
    const bool in = KC ? gr < R : gk < kend;
    const int n = in ? max(0, min(8, left)) : 0;
    const __nv_bfloat16 *g = n > 0 ? src + (KC ? (long long)gr * ld + gk : (long long)gk * ld + gr) : src;
    __nv_bfloat16 *d = tile + (KC ? r * GLD_K + k : k * GLD_R + r);
    if (vec) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(d)), "l"(g),
                   "r"(2 * n)
                   : "memory");
    } else {
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const uint32_t lo = 2 * e < n ? __bfloat16_as_ushort(g[2 * e]) : 0u;
        const uint32_t hi = 2 * e + 1 < n ? __bfloat16_as_ushort(g[2 * e + 1]) : 0u;
        w[e] = lo | (hi << 16);
      }
      *reinterpret_cast<uint4 *>(d) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

template <bool TA, bool TB>
__global__ void __launch_bounds__(128) gemm_bf16(int M, int N, int K, const __nv_bfloat16 *__restrict__ A, int lda,
                                                 const __nv_bfloat16 *__restrict__ B, int ldb, float *__restrict__ C,
                                                 int ldc) {
  __shared__ __align__(16) __nv_bfloat16 As[GST][GTILE], Bs[GST][GTILE];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.y * GBM, n0 = blockIdx.x * GBN;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  const int nk = (K + GBK - 1) / GBK;
  const bool va = (lda % 8) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  const bool vb = (ldb % 8) == 0 && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
  auto stage = [&](int c) {
    if (c < nk) {
      stage_tile<!TA>(As[c % GST], A, lda, m0, M, c * GBK, K, va);
      stage_tile<TB>(Bs[c % GST], B, ldb, n0, N, c * GBK, K, vb);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int c = 0; c < GST - 1; c++) stage(c);
  float acc[2][4][4] = {};
  for (int c = 0; c < nk; c++) {
    asm volatile("cp.async.wait_group %0;" ::"n"(GST - 2) : "memory");
    __syncthreads();  // tile c has landed for every thread, and all are done with the slot refilled next
    stage(c + GST - 1);
    const __nv_bfloat16 *a_s = As[c % GST], *b_s = Bs[c % GST];
#pragma unroll
    for (int ks = 0; ks < GBK; ks += 16) {
      uint32_t af[2][4], bp[2][4];
#pragma unroll
      for (int i = 0; i < 2; i++) {
        const int r = wm + 16 * i, lo = lane & 7, mid = ((lane >> 3) & 1) * 8, hi = (lane >> 4) * 8;
        ldsm4<TA>(af[i], TA ? a_s + (ks + lo + hi) * GLD_R + r + mid : a_s + (r + lo + mid) * GLD_K + ks + hi);
      }
#pragma unroll
      for (int j = 0; j < 2; j++) {  // 16 columns: two 8-column fragments
        const int r = wn + 16 * j, lo = lane & 7, mid = ((lane >> 3) & 1) * 8, hi = (lane >> 4) * 8;
        ldsm4<!TB>(bp[j], TB ? b_s + (r + lo + hi) * GLD_K + ks + mid : b_s + (ks + lo + mid) * GLD_R + r + hi);
      }
#pragma unroll
      for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const uint32_t bf[2] = {bp[j >> 1][(j & 1) * 2], bp[j >> 1][(j & 1) * 2 + 1]};
          mma_bf16(acc[i][j], af[i], bf);
        }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const int m = m0 + wm + 16 * i + g + (e >= 2 ? 8 : 0);
        const int n = n0 + wn + 8 * j + 2 * t + (e & 1);
        if (m < M && n < N) C[(long long)m * ldc + n] = acc[i][j][e];
      }
}

static cudaError_t gemm_mma(bool ta, bool tb, int M, int N, int K, const __nv_bfloat16 *A, int lda,
                            const __nv_bfloat16 *B, int ldb, float *C, int ldc, cudaStream_t s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  dim3 grd((N + GBN - 1) / GBN, (M + GBM - 1) / GBM);
  if (!ta && !tb) gemm_bf16<false, false><<<grd, 128, 0, s>>>(M, N, K, A, lda, B, ldb, C, ldc);
  else if (!ta && tb) gemm_bf16<false, true><<<grd, 128, 0, s>>>(M, N, K, A, lda, B, ldb, C, ldc);
  else if (ta && !tb) gemm_bf16<true, false><<<grd, 128, 0, s>>>(M, N, K, A, lda, B, ldb, C, ldc);
  else gemm_bf16<true, true><<<grd, 128, 0, s>>>(M, N, K, A, lda, B, ldb, C, ldc);
  return cudaGetLastError();
}

// Path of a GEMM: products with at least 128 rows run on the tcgen05 kernel
// (gemm_tc.cu: 128 x 128 tiles, accumulator in tensor memory); the narrow
// ones (weight gradients: rows = channels) on the mma.sync kernel above.
// path: 0 = by shape, 1 = mma.sync, 2 = tcgen05.
static cudaError_t gemm_path(int path, bool ta, bool tb, int M, int N, int K, const __nv_bfloat16 *A, int lda,
                             const __nv_bfloat16 *B, int ldb, float *C, int ldc, cudaStream_t s) {
  const bool tc = path == 2 || (path == 0 && M >= 128);
  return tc ? gemm_tcgen05(ta, tb, M, N, K, A, lda, B, ldb, C, ldc, s)
            : gemm_mma(ta, tb, M, N, K, A, lda, B, ldb, C, ldc, s);
}

static cudaError_t gemm(bool ta, bool tb, int M, int N, int K, const __nv_bfloat16 *A, int lda,
                        const __nv_bfloat16 *B, int ldb, float *C, int ldc, cudaStream_t s) {
  return gemm_path(0, ta, tb, M, N, K, A, lda, B, ldb, C, ldc, s);
}

// Weight gradients C[M x N] = A^T B, A [K][M], B [K][N] row-major with K =
// batch x length (up to 131072) and M, N the channels (16 .. 64, 8 .. 256):
// one output tile, a very long K.  The sum keeps its order (one chain of MMAs
// per element, ascending K), so what bounds the kernel is the chain, K / 16
// dependent mma.sync.  Therefore one m16n8 tile per warp (16 x 32 per block,
// as many chains side by side as the product has), nothing in the chain but
// the mma (each 32-row round's fragments are loaded during the round before),
// and three stages of 256 K rows of cp.async ahead of it.  16 x 8 over K =
// 65536: 0.18 ms, 43 ns per MMA, against 8.3 ms on the 64 x 64 tile kernel
// staged with 2-byte loads.
constexpr int WG_M = 16, WG_N = 32, WG_K = 256, WG_ST = 4;
constexpr int WG_LDA = WG_M + 8, WG_LDB = WG_N + 8;  // row pitches 48 and 80 bytes: ldmatrix rows in distinct banks
constexpr int WG_STAGE = WG_K * (WG_LDA + WG_LDB);   // elements
constexpr int WG_SMEM = WG_ST * WG_STAGE * 2;

__global__ void __launch_bounds__(128) gemm_wgrad(int M, int N, int K, const __nv_bfloat16 *__restrict__ A, int lda,
                                                  const __nv_bfloat16 *__restrict__ B, int ldb, float *__restrict__ C,
                                                  int ldc) {
  extern __shared__ __align__(16) __nv_bfloat16 sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.y * WG_M, n0 = blockIdx.x * WG_N;
  const int nk = (K + WG_K - 1) / WG_K;
  auto copy = [&](__nv_bfloat16 *d, const __nv_bfloat16 *base, int ld, int k, int c, int cols) {
    const int n = k < K ? max(0, min(8, cols - c)) : 0;  // elements in range, the rest is zero
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(d)),
                 "l"(n > 0 ? base + (long long)k * ld + c : base), "r"(2 * n)
                 : "memory");
  };
  auto stage = [&](int c) {
    if (c < nk) {
      __nv_bfloat16 *a = sm + (c % WG_ST) * WG_STAGE, *b = a + WG_K * WG_LDA;
#pragma unroll
      for (int q = tid; q < WG_K * 2; q += 128) copy(a + (q >> 1) * WG_LDA + (q & 1) * 8, A, lda, c * WG_K + (q >> 1), m0 + (q & 1) * 8, M);
#pragma unroll
      for (int q = tid; q < WG_K * 4; q += 128) copy(b + (q >> 2) * WG_LDB + (q & 3) * 8, B, ldb, c * WG_K + (q >> 2), n0 + (q & 3) * 8, N);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int c = 0; c < WG_ST - 1; c++) stage(c);
  float acc[4] = {};
  for (int c = 0; c < nk; c++) {
    asm volatile("cp.async.wait_group %0;" ::"n"(WG_ST - 2) : "memory");
    __syncthreads();
    stage(c + WG_ST - 1);
    const __nv_bfloat16 *a = sm + (c % WG_ST) * WG_STAGE, *b = a + WG_K * WG_LDA + warp * 8;
    uint32_t af[2][2][4], bf[2][4];
    auto frags = [&](int r) {  // fragments of the 32 K rows of round r
      ldsm4<true>(bf[r & 1], b + (32 * r + lane) * WG_LDB);
#pragma unroll
      for (int h = 0; h < 2; h++)
        ldsm4<true>(af[r & 1][h], a + (32 * r + 16 * h + (lane & 7) + (lane >> 4) * 8) * WG_LDA + ((lane >> 3) & 1) * 8);
    };
    frags(0);
#pragma unroll
    for (int r = 0; r < WG_K / 32; r++) {
      if (r + 1 < WG_K / 32) frags(r + 1);
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const uint32_t bh[2] = {bf[r & 1][2 * h], bf[r & 1][2 * h + 1]};
        mma_bf16(acc, af[r & 1][h], bh);
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
  for (int e = 0; e < 4; e++) {
    const int m = m0 + (lane >> 2) + (e >= 2 ? 8 : 0), n = n0 + warp * 8 + 2 * (lane & 3) + (e & 1);
    if (m < M && n < N) C[(long long)m * ldc + n] = acc[e];
  }
}

// C = A^T B of the backward pass: gemm_wgrad where the rows are channels (M <
// 128, as gemm_path's narrow products), 16-byte aligned, and K is long enough
// for the stages to fill; otherwise by shape.
static cudaError_t gemm_grad(int M, int N, int K, const __nv_bfloat16 *A, int lda, const __nv_bfloat16 *B, int ldb,
                             float *C, cudaStream_t s) {
  const bool vec = lda % 8 == 0 && ldb % 8 == 0 && ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) == 0;
  if (M >= 128 || K < 2 * WG_K || !vec) return gemm(true, false, M, N, K, A, lda, B, ldb, C, N, s);
  cudaError_t e = cudaFuncSetAttribute(gemm_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, WG_SMEM);
  if (e != cudaSuccess) return e;
  gemm_wgrad<<<dim3((N + WG_N - 1) / WG_N, (M + WG_M - 1) / WG_M), 128, WG_SMEM, s>>>(M, N, K, A, lda, B, ldb, C, N);
  return cudaGetLastError();
}

// ------------------------------------------------------------ elementwise
__device__ __forceinline__ float gelu_f(float x) {
  const float u = 0.7978845608028654f * (x + 0.044715f * x * x * x);
  return 0.5f * x * (1.f + tanhf(u));
}
__device__ __forceinline__ float gelu_df(float x) {
  const float u = 0.7978845608028654f * (x + 0.044715f * x * x * x);
  const float th = tanhf(u);
  return 0.5f * (1.f + th) + 0.5f * x * (1.f - th * th) * 0.7978845608028654f * (1.f + 3.f * 0.044715f * x * x);
}

#define GRID_STRIDE(q, n) for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < (n); \
                               q += (long long)gridDim.x * blockDim.x)

__global__ void k_normalize(const float *X, const float *mean, const float *scale, int n, int d, __nv_bfloat16 *out) {
  GRID_STRIDE(q, (long long)n * d) out[q] = __float2bfloat16((X[q] - mean[q % d]) / scale[q % d]);
}

// pre = Z + bias (row-major [rows][N]), act = gelu(pre) as BF16
__global__ void k_bias_gelu(const float *Z, const float *bias, long long rows, int N, float *pre, __nv_bfloat16 *act) {
  GRID_STRIDE(q, rows * N) {
    const float v = Z[q] + bias[q % N];
    pre[q] = v;
    act[q] = __float2bfloat16(gelu_f(v));
  }
}

// y = Z + bias (final layer, FP32)
__global__ void k_bias(const float *Z, const float *bias, long long rows, int N, float *y) {
  GRID_STRIDE(q, rows * N) y[q] = Z[q] + bias[q % N];
}

// col2im of a transposed convolution (kernel 4, stride 2, padding 1):
// out[b][t][co] = bias[co] + sum over the taps (s, q) with 2 s - 1 + q = t of Z[b][s][co*4 + q]
__global__ void k_col2im(const float *Z, const float *bias, int B, int Lin, int Cout, float *pre,
                         __nv_bfloat16 *act) {
  const int Lout = 2 * Lin;
  GRID_STRIDE(q, (long long)B * Lout * Cout) {
    const int co = (int)(q % Cout);
    const long long bt = q / Cout;
    const int t = (int)(bt % Lout), b = (int)(bt / Lout);
    float v = bias[co];
    // t even: taps q = 1 (s = t/2), q = 3 (s = t/2 - 1); t odd: q = 0 (s = (t+1)/2), q = 2 (s = (t-1)/2)
    const int qa = (t & 1) ? 0 : 1, qb = qa + 2;
    const int sa = (t + 1 - qa) / 2, sb = (t + 1 - qb) / 2;
    if (sa >= 0 && sa < Lin) v += Z[((long long)b * Lin + sa) * (Cout * 4) + co * 4 + qa];
    if (sb >= 0 && sb < Lin) v += Z[((long long)b * Lin + sb) * (Cout * 4) + co * 4 + qb];
    pre[q] = v;
    act[q] = __float2bfloat16(gelu_f(v));
  }
}

// dz = da * gelu'(pre), FP32 and BF16 copies
__global__ void k_gelu_bwd(const float *da, const float *pre, long long n, float *dz, __nv_bfloat16 *dz16) {
  GRID_STRIDE(q, n) {
    const float v = da[q] * gelu_df(pre[q]);
    dz[q] = v;
    dz16[q] = __float2bfloat16(v);
  }
}

// Backward of one transposed convolution's activation: v[b][t][co] = da *
// gelu'(pre) and its im2col dZ[b][s][co*4+q] = v[b][2s-1+q][co] (BF16, zero
// outside), v itself in FP32 for the bias gradient.  One thread per (b, s, co)
// reads the four outputs its taps land on (each of them twice over the
// launch, the second time from L1) and writes its four dZ values as one
// 8-byte word, which saves the write and two reads of v a separate im2col made.
__global__ void k_conv_bwd(const float *__restrict__ da, const float *__restrict__ pre, int B, int Lin, int Cout,
                           float *__restrict__ dz, __nv_bfloat16 *__restrict__ dZ) {
  const int Lout = 2 * Lin;
  GRID_STRIDE(q, (long long)B * Lin * Cout) {
    const int co = (int)(q % Cout);
    const long long bs = q / Cout;
    const int s = (int)(bs % Lin), b = (int)(bs / Lin);
    __nv_bfloat16 h[4];
#pragma unroll
    for (int tap = 0; tap < 4; tap++) {
      const int t = 2 * s - 1 + tap;
      const long long o = ((long long)b * Lout + t) * Cout + co;
      float v = 0.f;
      if (t >= 0 && t < Lout) {
        v = da[o] * gelu_df(pre[o]);
        if (tap == 1 || tap == 2) dz[o] = v;
      }
      h[tap] = __float2bfloat16(v);
    }
    uint2 u;
    u.x = (uint32_t)__bfloat16_as_ushort(h[0]) | ((uint32_t)__bfloat16_as_ushort(h[1]) << 16);
    u.y = (uint32_t)__bfloat16_as_ushort(h[2]) | ((uint32_t)__bfloat16_as_ushort(h[3]) << 16);
    *reinterpret_cast<uint2 *>(dZ + 4 * q) = u;
  }
}

// Column sums of a [rows][N] FP32 matrix into out[N], in a fixed order: per
// column, sums over consecutive chunks of rows, then the sum of those.  Block
// = 128 threads over (column, chunk) pairs, column fastest, so that narrow
// matrices (8 .. 64 columns) still fill the warps; both loops keep 16 loads
// in flight ahead of their serial additions.
__global__ void __launch_bounds__(128) k_colsum_partial(const float *X, long long rows, int N, int chunk, int parts,
                                                        float *part) {
  const long long q = blockIdx.x * 128LL + threadIdx.x;
  if (q >= (long long)N * parts) return;
  const int n = (int)(q % N);
  const long long r0 = q / N * chunk, r1 = min(rows, r0 + chunk);
  float acc = 0.f;
  long long r = r0;
  for (; r + 16 <= r1; r += 16) {
    float v[16];
#pragma unroll
    for (int e = 0; e < 16; e++) v[e] = X[(r + e) * N + n];
#pragma unroll
    for (int e = 0; e < 16; e++) acc += v[e];
  }
  for (; r < r1; r++) acc += X[r * N + n];
  part[q] = acc;
}
__global__ void __launch_bounds__(32) k_colsum_final(const float *part, int parts, int N, float *out) {
  const int n = blockIdx.x * 32 + threadIdx.x;
  if (n >= N) return;
  float acc = 0.f;
  int p = 0;
  for (; p + 16 <= parts; p += 16) {
    float v[16];
#pragma unroll
    for (int e = 0; e < 16; e++) v[e] = part[(long long)(p + e) * N + n];
#pragma unroll
    for (int e = 0; e < 16; e++) acc += v[e];
  }
  for (; p < parts; p++) acc += part[(long long)p * N + n];
  out[n] = acc;
}

// MSE of channels-last predictions y[b][t][c] against targets T[b][c][t]:
// loss partials per block, gradient dy = 2 (y - T) / count
__global__ void k_mse(const float *y, const float *T, int B, int L, int Cc, float inv_count, float inv_ys, float *dy,
                      __nv_bfloat16 *dy16, float *loss_part) {
  __shared__ float red[256];
  float acc = 0.f;
  GRID_STRIDE(q, (long long)B * L * Cc) {
    const int c = (int)(q % Cc);
    const long long bt = q / Cc;
    const int t = (int)(bt % L), b = (int)(bt / L);
    const float e = y[q] - T[((long long)b * Cc + c) * L + t] * inv_ys;
    const float d = 2.f * e * inv_count;
    dy[q] = d;
    dy16[q] = __float2bfloat16(d);
    acc += e * e;
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) loss_part[blockIdx.x] = red[0];
}

// channels-last [b][t][c] -> [b][c][t]
__global__ void k_to_channels_first(const float *y, int B, int L, int Cc, float scale, float *out) {
  GRID_STRIDE(q, (long long)B * L * Cc) {
    const int t = (int)(q % L);
    const long long bc = q / L;
    const int c = (int)(bc % Cc), b = (int)(bc / Cc);
    out[q] = y[((long long)b * L + t) * Cc + c] * scale;
  }
}

__global__ void k_to_bf16(const float *x, long long n, __nv_bfloat16 *y) {
  GRID_STRIDE(q, n) y[q] = __float2bfloat16(x[q]);
}

__global__ void k_adam(float *w, const float *g, float *m, float *v, __nv_bfloat16 *w16, long long n, float lr,
                       float b1, float b2, float eps, float c1, float c2) {
  GRID_STRIDE(q, n) {
    const float gq = g[q];
    const float mq = b1 * m[q] + (1.f - b1) * gq, vq = b2 * v[q] + (1.f - b2) * gq * gq;
    m[q] = mq;
    v[q] = vq;
    const float wq = w[q] - lr * (mq / c1) / (sqrtf(vq / c2) + eps);
    w[q] = wq;
    w16[q] = __float2bfloat16(wq);
  }
}

// per case b: num[b] = sum (y - y0)^2 and den[b] = sum y0^2 over its `per`
// outputs (one block per case, fixed-order tree in the block)
__global__ void __launch_bounds__(256) k_diff_norms(const float *y, const float *y0, long long per, float *num,
                                                    float *den) {
  const long long o = (long long)blockIdx.x * per;
  float a = 0.f, b = 0.f;
  for (long long q = threadIdx.x; q < per; q += 256) {
    const float u = y0[o + q], d = y[o + q] - u;
    a += d * d;
    b += u * u;
  }
  __shared__ float sa[256], sb[256];
  sa[threadIdx.x] = a;
  sb[threadIdx.x] = b;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sa[threadIdx.x] += sa[threadIdx.x + w];
      sb[threadIdx.x] += sb[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    num[blockIdx.x] = sa[0];
    den[blockIdx.x] = sb[0];
  }
}

// gather rows of the device training set into a minibatch
__global__ void k_gather(const float *src, const int *idx, int n, long long row, float *dst) {
  GRID_STRIDE(q, (long long)n * row) dst[q] = src[(long long)idx[q / row] * row + q % row];
}

static int egrid(long long n) { return (int)std::min<long long>((n + 255) / 256, 152 * 16); }

}  // namespace cwell

// ======================================================================= host
using namespace cwell;

constexpr int COLSUM_PARTS = 4096;  // at most this many row chunks per column sum
constexpr int LOSS_PARTS = 1024;    // blocks of the loss kernel
constexpr int LOSS_KEEP = 1024;     // minibatches whose loss partials training keeps on the device (4 MB)

struct sur_s {
  sur_cfg_t cfg{};
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  int device = 0;
  long long nparam = 0;
  int max_batch = 0;
  std::vector<long long> off;  // parameter offsets: W1 b1 W2 b2 W3 b3 (T_l t_l)*nup Wf bf
  std::vector<int> chans;      // C0, C1, ..., C_nup
  float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
  __nv_bfloat16 *w16 = nullptr;
  float *x_mean = nullptr, *x_scale = nullptr;
  float y_scale = 1.f;  // outputs are y_scale times the network's (normalised) output
  long long adam_t = 0;
  // activations (sized for max_batch)
  std::vector<float *> pre;             // per layer pre-activations (FP32)
  std::vector<__nv_bfloat16 *> act;     // per layer activations (BF16), act[0] = normalised input
  float *z = nullptr, *y = nullptr, *dy = nullptr, *da = nullptr, *dz = nullptr, *part = nullptr, *lossp = nullptr;
  __nv_bfloat16 *dy16 = nullptr;
  // backward: per layer the gradient of its pre-activation (FP32) and the BF16 operand of its weight gradient
  std::vector<float *> gz;
  std::vector<__nv_bfloat16 *> gz16;
  // The weight and bias gradients hang off the chain of data gradients and
  // are themselves long serial sums, so they run beside it: side[0] the bias
  // sums, side[1] the last layer's weight gradient (the longest), side[2] the
  // others.  ready[q] marks operand q on the handle's stream, done[k] the end
  // of side[k]; the handle's stream waits for all of them before a backward
  // pass returns.
  static constexpr int SIDES = 3, MAX_READY = 12;
  cudaStream_t side[SIDES] = {};
  cudaEvent_t done[SIDES] = {}, ready[MAX_READY] = {};
  float *xb = nullptr, *tb = nullptr;
  std::vector<void *> allocs;
  std::vector<float> gate_x, gate_err;  // normalised validation inputs and their errors
  std::string err;
};

static thread_local std::string g_sur_err;
static int sfail(sur_t *s, int code, const std::string &m);

// a bounded wait of the tcgen05 GEMM that gave up surfaces as SIM_ETIMEOUT
static int tc_status(sur_t *s) {
  int st = 0;
  cudaError_t e = gemm_tcgen05_status(&st, s->stream);
  if (e != cudaSuccess) return sfail(s, SIM_ECUDA, cudaGetErrorString(e));
  if (st) return sfail(s, SIM_ETIMEOUT, "a tcgen05 GEMM wait gave up");
  return SIM_OK;
}

static int sfail(sur_t *s, int code, const std::string &m) {
  if (s) s->err = m;
  else g_sur_err = m;
  return code;
}

#define SCK(s, call)                                                                            \
  do {                                                                                          \
    cudaError_t e_ = (call);                                                                    \
    if (e_ != cudaSuccess) return sfail(s, SIM_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

template <typename P>
static int salloc(sur_t *s, P **p, size_t bytes) {
  cudaError_t e = cudaMalloc((void **)p, std::max<size_t>(bytes, 16));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return sfail(s, SIM_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  }
  s->allocs.push_back(*p);
  return SIM_OK;
}

static int L_out(const sur_t *s) { return s->cfg.l0 << s->cfg.n_up; }

// layer widths: dense sizes and per-layer activation element counts
static void layout(sur_t *s) {
  const sur_cfg_t &c = s->cfg;
  s->chans.assign(c.chans, c.chans + c.n_up + 1);
  s->off.clear();
  long long o = 0;
  auto add = [&](long long n) {
    s->off.push_back(o);
    o += n;
  };
  add((long long)c.in_dim * c.h1);
  add(c.h1);
  add((long long)c.h1 * c.h2);
  add(c.h2);
  add((long long)c.h2 * c.l0 * c.chans[0]);
  add((long long)c.l0 * c.chans[0]);
  for (int l = 0; l < c.n_up; l++) {
    add((long long)c.chans[l] * c.chans[l + 1] * 4);
    add(c.chans[l + 1]);
  }
  add((long long)c.chans[c.n_up] * c.out_ch);
  add(c.out_ch);
  s->off.push_back(o);
  s->nparam = o;
}

static void release_side(sur_t *s) {
  for (cudaStream_t x : s->side)
    if (x) cudaStreamDestroy(x);
  for (cudaEvent_t x : s->done)
    if (x) cudaEventDestroy(x);
  for (cudaEvent_t x : s->ready)
    if (x) cudaEventDestroy(x);
}

extern "C" int sur_create(const sur_cfg_t *cfg, const sim_opts_t *opts, sur_t **out) {
  if (!out) return sfail(nullptr, SIM_EINVAL, "out is null");
  *out = nullptr;
  if (!cfg || cfg->in_dim < 1 || cfg->h1 < 1 || cfg->h2 < 1 || cfg->l0 < 1 || cfg->n_up < 0 || cfg->n_up > 8 ||
      cfg->out_ch < 1 || cfg->max_batch < 1)
    return sfail(nullptr, SIM_EINVAL, "bad surrogate configuration");
  for (int l = 0; l <= cfg->n_up; l++)
    if (cfg->chans[l] < 1) return sfail(nullptr, SIM_EINVAL, "bad channel count");
  sur_t *s = new sur_t();
  s->cfg = *cfg;
  s->max_batch = cfg->max_batch;
  s->device = opts ? opts->device : 0;
  auto bail = [&](int rc) {
    g_sur_err = s->err;
    release_side(s);
    for (void *p : s->allocs) cudaFree(p);
    if (s->own_stream) cudaStreamDestroy(s->stream);
    delete s;
    return rc;
  };
  cudaError_t e = cudaSetDevice(s->device);
  if (e != cudaSuccess) return bail(sfail(s, SIM_ECUDA, cudaGetErrorString(e)));
  if (opts && opts->cuda_stream) {
    s->stream = (cudaStream_t)opts->cuda_stream;
  } else {
    if ((e = cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking)) != cudaSuccess)
      return bail(sfail(s, SIM_ECUDA, cudaGetErrorString(e)));
    s->own_stream = true;
  }
  for (int k = 0; k < sur_t::SIDES && e == cudaSuccess; k++)
    if ((e = cudaStreamCreateWithFlags(&s->side[k], cudaStreamNonBlocking)) == cudaSuccess)
      e = cudaEventCreateWithFlags(&s->done[k], cudaEventDisableTiming);
  for (int k = 0; k < sur_t::MAX_READY && e == cudaSuccess; k++)
    e = cudaEventCreateWithFlags(&s->ready[k], cudaEventDisableTiming);
  if (e != cudaSuccess) return bail(sfail(s, SIM_ECUDA, cudaGetErrorString(e)));
  layout(s);
  const long long P = s->nparam;
  int rc;
  if ((rc = salloc(s, &s->w, P * 4)) || (rc = salloc(s, &s->g, P * 4)) || (rc = salloc(s, &s->m, P * 4)) ||
      (rc = salloc(s, &s->v, P * 4)) || (rc = salloc(s, &s->w16, P * 2)) || (rc = salloc(s, &s->x_mean, cfg->in_dim * 4)) ||
      (rc = salloc(s, &s->x_scale, cfg->in_dim * 4)))
    return bail(rc);
  const int B = s->max_batch, Lf = L_out(s);
  // activations: layer 0 input, 1 h1, 2 h2, 3 a0 (= reshaped dense), 4.. convT outputs
  std::vector<long long> an = {(long long)B * cfg->in_dim, (long long)B * cfg->h1, (long long)B * cfg->h2,
                               (long long)B * cfg->l0 * cfg->chans[0]};
  long long zmax = std::max<long long>((long long)B * cfg->l0 * cfg->chans[0], (long long)B * Lf * cfg->out_ch);
  for (int l = 0; l < cfg->n_up; l++) {
    const long long Lin = (long long)cfg->l0 << l;
    an.push_back((long long)B * 2 * Lin * cfg->chans[l + 1]);
    zmax = std::max(zmax, (long long)B * Lin * cfg->chans[l + 1] * 4);
  }
  long long amax = 0;
  for (long long a : an) amax = std::max(amax, a);
  zmax = std::max(zmax, amax);
  s->pre.resize(an.size());
  s->act.resize(an.size());
  s->gz.resize(an.size());
  s->gz16.resize(an.size());
  for (size_t l = 0; l < an.size(); l++) {
    if ((rc = salloc(s, &s->pre[l], an[l] * 4)) || (rc = salloc(s, &s->act[l], an[l] * 2))) return bail(rc);
    // a convolution's dZ has two values per output (four taps, half as many inputs)
    if (l > 0 && ((rc = salloc(s, &s->gz[l], an[l] * 4)) || (rc = salloc(s, &s->gz16[l], an[l] * (l > 3 ? 4 : 2)))))
      return bail(rc);
  }
  if ((rc = salloc(s, &s->z, zmax * 4)) || (rc = salloc(s, &s->y, (long long)B * Lf * cfg->out_ch * 4)) ||
      (rc = salloc(s, &s->dy, (long long)B * Lf * cfg->out_ch * 4)) || (rc = salloc(s, &s->da, zmax * 4)) ||
      (rc = salloc(s, &s->dz, (long long)B * Lf * cfg->out_ch * 4)) ||
      (rc = salloc(s, &s->dy16, (long long)B * Lf * cfg->out_ch * 2)) ||
      (rc = salloc(s, &s->part, (long long)COLSUM_PARTS * COLSUM_PARTS * 4)) ||
      (rc = salloc(s, &s->lossp, LOSS_PARTS * 4)) || (rc = salloc(s, &s->xb, (long long)B * cfg->in_dim * 4)) ||
      (rc = salloc(s, &s->tb, (long long)B * Lf * cfg->out_ch * 4)))
    return bail(rc);
  // initial weights: uniform +-sqrt(6 / (fan_in + fan_out)) from SplitMix64, biases 0
  std::vector<float> w(P, 0.f);
  uint64_t st = cfg->seed;
  auto uni = [&]() {
    uint64_t z = (st += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
  };
  auto fill = [&](int slot, double fan_in, double fan_out) {
    const double a = sqrt(6.0 / (fan_in + fan_out));
    for (long long q = s->off[slot]; q < s->off[slot + 1]; q++) w[q] = (float)((2.0 * uni() - 1.0) * a);
  };
  fill(0, cfg->in_dim, cfg->h1);
  fill(2, cfg->h1, cfg->h2);
  fill(4, cfg->h2, (double)cfg->l0 * cfg->chans[0]);
  for (int l = 0; l < cfg->n_up; l++) fill(6 + 2 * l, 2.0 * cfg->chans[l], 2.0 * cfg->chans[l + 1]);
  fill(6 + 2 * cfg->n_up, cfg->chans[cfg->n_up], cfg->out_ch);
  std::vector<float> ones(cfg->in_dim, 1.f), zeros(cfg->in_dim, 0.f);
  if ((e = cudaMemcpy(s->w, w.data(), P * 4, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemcpy(s->x_mean, zeros.data(), cfg->in_dim * 4, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemcpy(s->x_scale, ones.data(), cfg->in_dim * 4, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemset(s->m, 0, P * 4)) != cudaSuccess || (e = cudaMemset(s->v, 0, P * 4)) != cudaSuccess)
    return bail(sfail(s, SIM_ECUDA, cudaGetErrorString(e)));
  k_to_bf16<<<egrid(P), 256, 0, s->stream>>>(s->w, P, s->w16);
  if ((e = cudaStreamSynchronize(s->stream)) != cudaSuccess) return bail(sfail(s, SIM_ECUDA, cudaGetErrorString(e)));
  *out = s;
  return SIM_OK;
}

static float *Wp(sur_t *s, int slot) { return s->w + s->off[slot]; }
static __nv_bfloat16 *W16(sur_t *s, int slot) { return s->w16 + s->off[slot]; }
static float *Gp(sur_t *s, int slot) { return s->g + s->off[slot]; }

static cudaError_t colsum(const float *X, long long rows, int N, float *out, float *part, cudaStream_t st) {
  const int chunk = 256;
  const int parts = (int)std::min<long long>((rows + chunk - 1) / chunk, COLSUM_PARTS);
  const int ch = (int)((rows + parts - 1) / parts);
  k_colsum_partial<<<(int)(((long long)N * parts + 127) / 128), 128, 0, st>>>(X, rows, N, ch, parts, part);
  k_colsum_final<<<(N + 31) / 32, 32, 0, st>>>(part, parts, N, out);
  return cudaGetLastError();
}

// forward pass of n <= max_batch samples whose raw inputs are in s->xb
static cudaError_t forward(sur_t *s, int n) {
  const sur_cfg_t &c = s->cfg;
  cudaStream_t st = s->stream;
  cudaError_t e;
  k_normalize<<<egrid((long long)n * c.in_dim), 256, 0, st>>>(s->xb, s->x_mean, s->x_scale, n, c.in_dim, s->act[0]);
  const int dims[4] = {c.in_dim, c.h1, c.h2, c.l0 * c.chans[0]};
  for (int l = 0; l < 3; l++) {
    if ((e = gemm(false, false, n, dims[l + 1], dims[l], s->act[l], dims[l], W16(s, 2 * l), dims[l + 1], s->z,
                  dims[l + 1], st)) != cudaSuccess)
      return e;
    k_bias_gelu<<<egrid((long long)n * dims[l + 1]), 256, 0, st>>>(s->z, Wp(s, 2 * l + 1), n, dims[l + 1],
                                                                     s->pre[l + 1], s->act[l + 1]);
  }
  for (int l = 0; l < c.n_up; l++) {
    const int Lin = c.l0 << l, Cin = c.chans[l], Cout = c.chans[l + 1];
    const long long rows = (long long)n * Lin;
    if ((e = gemm(false, false, (int)rows, Cout * 4, Cin, s->act[3 + l], Cin, W16(s, 6 + 2 * l), Cout * 4, s->z,
                  Cout * 4, st)) != cudaSuccess)
      return e;
    k_col2im<<<egrid(rows * 2 * Cout), 256, 0, st>>>(s->z, Wp(s, 7 + 2 * l), n, Lin, Cout, s->pre[4 + l],
                                                      s->act[4 + l]);
  }
  const int Lf = L_out(s), Cl = c.chans[c.n_up];
  const long long rows = (long long)n * Lf;
  if ((e = gemm(false, false, (int)rows, c.out_ch, Cl, s->act[3 + c.n_up], Cl, W16(s, 6 + 2 * c.n_up), c.out_ch,
                s->z, c.out_ch, st)) != cudaSuccess)
    return e;
  k_bias<<<egrid(rows * c.out_ch), 256, 0, st>>>(s->z, Wp(s, 7 + 2 * c.n_up), rows, c.out_ch, s->y);
  return cudaGetLastError();
}

// the handle's stream waits for what the side streams hold (the host does where
// that cannot be enqueued)
static cudaError_t join_sides(sur_t *s) {
  cudaError_t first = cudaSuccess;
  for (int k = 0; k < sur_t::SIDES; k++) {
    cudaError_t e = cudaEventRecord(s->done[k], s->side[k]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s->stream, s->done[k], 0);
    if (e != cudaSuccess) cudaStreamSynchronize(s->side[k]);
    if (first == cudaSuccess) first = e;
  }
  return first;
}

static cudaError_t enqueue_backward(sur_t *s, int n, float *lossp) {
  const sur_cfg_t &c = s->cfg;
  cudaStream_t st = s->stream;
  cudaError_t e = cudaSuccess;
  const int Lf = L_out(s), Cl = c.chans[c.n_up];
  const long long rows = (long long)n * Lf, count = rows * c.out_ch;
  int nready = 0;
  // weight and bias gradient of one layer, operands just enqueued on st:
  // dW[M x N] = A^T D over K rows, db = column sums of d (drows x N2)
  auto grads = [&](int side, int M, int N, int K, const __nv_bfloat16 *A, const __nv_bfloat16 *D, float *dW,
                   const float *d, long long drows, int N2, float *db) {
    cudaEvent_t r = s->ready[nready++];
    if ((e = cudaEventRecord(r, st)) != cudaSuccess) return e;
    for (int k : {0, side})
      if ((e = cudaStreamWaitEvent(s->side[k], r, 0)) != cudaSuccess) return e;
    if ((e = colsum(d, drows, N2, db, s->part, s->side[0])) != cudaSuccess) return e;
    return e = gemm_grad(M, N, K, A, M, D, N, dW, s->side[side]);
  };
  // data gradient: s->da = D W^T
  auto data = [&](int M, int N, int K, const __nv_bfloat16 *D, const __nv_bfloat16 *W) {
    return e = gemm(false, true, M, N, K, D, K, W, K, s->da, N, st);
  };
  k_mse<<<LOSS_PARTS, 256, 0, st>>>(s->y, s->tb, n, Lf, c.out_ch, 1.f / (float)count, 1.f / s->y_scale, s->dy, s->dy16,
                                    lossp);
  // final 1x1 layer
  if (grads(1, Cl, c.out_ch, (int)rows, s->act[3 + c.n_up], s->dy16, Gp(s, 6 + 2 * c.n_up), s->dy, rows, c.out_ch,
            Gp(s, 7 + 2 * c.n_up)) != cudaSuccess)
    return e;
  if (data((int)rows, Cl, c.out_ch, s->dy16, W16(s, 6 + 2 * c.n_up)) != cudaSuccess) return e;
  // transposed convolutions, last to first
  for (int l = c.n_up - 1; l >= 0; l--) {
    const int Lin = c.l0 << l, Cin = c.chans[l], Cout = c.chans[l + 1];
    const long long irow = (long long)n * Lin;
    k_conv_bwd<<<egrid(irow * Cout), 256, 0, st>>>(s->da, s->pre[4 + l], n, Lin, Cout, s->gz[4 + l], s->gz16[4 + l]);
    if (grads(2, Cin, Cout * 4, (int)irow, s->act[3 + l], s->gz16[4 + l], Gp(s, 6 + 2 * l), s->gz[4 + l], 2 * irow,
              Cout, Gp(s, 7 + 2 * l)) != cudaSuccess)
      return e;
    if (data((int)irow, Cin, Cout * 4, s->gz16[4 + l], W16(s, 6 + 2 * l)) != cudaSuccess) return e;
  }
  // dense layers 3, 2, 1
  const int dims[4] = {c.in_dim, c.h1, c.h2, c.l0 * c.chans[0]};
  for (int l = 2; l >= 0; l--) {
    const long long nel = (long long)n * dims[l + 1];
    k_gelu_bwd<<<egrid(nel), 256, 0, st>>>(s->da, s->pre[l + 1], nel, s->gz[l + 1], s->gz16[l + 1]);
    if (grads(2, dims[l], dims[l + 1], n, s->act[l], s->gz16[l + 1], Gp(s, 2 * l), s->gz[l + 1], n, dims[l + 1],
              Gp(s, 2 * l + 1)) != cudaSuccess)
      return e;
    if (l > 0 && data(n, dims[l], dims[l + 1], s->gz16[l + 1], W16(s, 2 * l)) != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

// Gradient into s->g and the loss kernel's LOSS_PARTS partial sums into lossp
// (device), for the targets in s->tb.  The handle's stream ends behind all of it,
// also after a failure: what was enqueued by then still writes s->g and reads the
// activations the next call overwrites.
static cudaError_t backward(sur_t *s, int n, float *lossp) {
  const cudaError_t e = enqueue_backward(s, n, lossp), j = join_sides(s);
  return e != cudaSuccess ? e : j;
}

// the loss from the partial sums of a minibatch of n samples
static float loss_of(const sur_t *s, const float *parts, int n) {
  double acc = 0;
  for (int q = 0; q < LOSS_PARTS; q++) acc += parts[q];
  return (float)(acc / ((double)n * L_out(s) * s->cfg.out_ch));
}

extern "C" int sur_param_count(const sur_t *s, long long *n) {
  if (!s || !n) return SIM_EINVAL;
  *n = s->nparam;
  return SIM_OK;
}

extern "C" int sur_get_params(sur_t *s, float *out, size_t n) {
  if (!s || !out || n < (size_t)s->nparam) return s ? sfail(s, SIM_EINVAL, "buffer too small") : SIM_EINVAL;
  SCK(s, cudaStreamSynchronize(s->stream));
  SCK(s, cudaMemcpy(out, s->w, s->nparam * 4, cudaMemcpyDeviceToHost));
  return SIM_OK;
}

extern "C" int sur_set_params(sur_t *s, const float *in, size_t n) {
  if (!s || !in || n < (size_t)s->nparam) return s ? sfail(s, SIM_EINVAL, "buffer too small") : SIM_EINVAL;
  SCK(s, cudaStreamSynchronize(s->stream));
  SCK(s, cudaMemcpy(s->w, in, s->nparam * 4, cudaMemcpyHostToDevice));
  k_to_bf16<<<egrid(s->nparam), 256, 0, s->stream>>>(s->w, s->nparam, s->w16);
  SCK(s, cudaGetLastError());
  SCK(s, cudaMemset(s->m, 0, s->nparam * 4));
  SCK(s, cudaMemset(s->v, 0, s->nparam * 4));
  s->adam_t = 0;
  return SIM_OK;
}

extern "C" int sur_set_normalization(sur_t *s, const float *x_mean, const float *x_scale, float y_scale) {
  if (!s || !x_mean || !x_scale) return SIM_EINVAL;
  if (!(y_scale > 0) || !isfinite(y_scale)) return sfail(s, SIM_EINVAL, "output scale must be positive and finite");
  s->y_scale = y_scale;
  SCK(s, cudaStreamSynchronize(s->stream));
  for (int q = 0; q < s->cfg.in_dim; q++)
    if (!(x_scale[q] != 0.f) || !isfinite(x_scale[q]) || !isfinite(x_mean[q]))
      return sfail(s, SIM_EINVAL, "normalisation scales must be finite and non-zero");
  SCK(s, cudaMemcpy(s->x_mean, x_mean, s->cfg.in_dim * 4, cudaMemcpyHostToDevice));
  SCK(s, cudaMemcpy(s->x_scale, x_scale, s->cfg.in_dim * 4, cudaMemcpyHostToDevice));
  return SIM_OK;
}

extern "C" int sur_forward(sur_t *s, const float *X, int n, float *Y) {
  if (!s || n < 0 || (n > 0 && (!X || !Y))) return s ? sfail(s, SIM_EINVAL, "bad arguments") : SIM_EINVAL;
  SCK(s, cudaSetDevice(s->device));
  const sur_cfg_t &c = s->cfg;
  const int Lf = L_out(s);
  for (int b0 = 0; b0 < n; b0 += s->max_batch) {
    const int nb = std::min(s->max_batch, n - b0);
    SCK(s, cudaMemcpyAsync(s->xb, X + (size_t)b0 * c.in_dim, (size_t)nb * c.in_dim * 4, cudaMemcpyHostToDevice,
                           s->stream));
    SCK(s, forward(s, nb));
    k_to_channels_first<<<egrid((long long)nb * Lf * c.out_ch), 256, 0, s->stream>>>(s->y, nb, Lf, c.out_ch,
                                                                                     s->y_scale, s->dz);
    SCK(s, cudaGetLastError());
    SCK(s, cudaMemcpyAsync(Y + (size_t)b0 * Lf * c.out_ch, s->dz, (size_t)nb * Lf * c.out_ch * 4,
                           cudaMemcpyDeviceToHost, s->stream));
  }
  SCK(s, cudaStreamSynchronize(s->stream));
  return tc_status(s);
}

extern "C" int sur_sensitivity(sur_t *s, const float *X, int n, float step, float *sens) {
  if (!s || n < 0 || (n > 0 && (!X || !sens)) || !(step > 0.f))
    return s ? sfail(s, SIM_EINVAL, "bad arguments") : SIM_EINVAL;
  SCK(s, cudaSetDevice(s->device));
  const sur_cfg_t &c = s->cfg;
  const long long per = (long long)L_out(s) * c.out_ch;
  std::vector<float> scale(c.in_dim), xp((size_t)s->max_batch * c.in_dim), num(s->max_batch), den(s->max_batch);
  SCK(s, cudaMemcpy(scale.data(), s->x_scale, c.in_dim * 4, cudaMemcpyDeviceToHost));
  float *nd = s->part;  // [2][max_batch] partial norms (the column-sum scratch, idle here)
  for (int b0 = 0; b0 < n; b0 += s->max_batch) {
    const int nb = std::min(s->max_batch, n - b0);
    const float *xc = X + (size_t)b0 * c.in_dim;
    SCK(s, cudaMemcpyAsync(s->xb, xc, (size_t)nb * c.in_dim * 4, cudaMemcpyHostToDevice, s->stream));
    SCK(s, forward(s, nb));
    SCK(s, cudaMemcpyAsync(s->dy, s->y, (size_t)nb * per * 4, cudaMemcpyDeviceToDevice, s->stream));
    for (int q = 0; q < nb; q++) sens[b0 + q] = 0.f;
    for (int d = 0; d < c.in_dim; d++) {
      // the input moved by `step` in normalised units along dimension d
      for (int q = 0; q < nb; q++)
        for (int e = 0; e < c.in_dim; e++)
          xp[(size_t)q * c.in_dim + e] = xc[(size_t)q * c.in_dim + e] + (e == d ? step * scale[d] : 0.f);
      SCK(s, cudaMemcpyAsync(s->xb, xp.data(), (size_t)nb * c.in_dim * 4, cudaMemcpyHostToDevice, s->stream));
      SCK(s, forward(s, nb));
      k_diff_norms<<<nb, 256, 0, s->stream>>>(s->y, s->dy, per, nd, nd + s->max_batch);
      SCK(s, cudaGetLastError());
      SCK(s, cudaMemcpyAsync(num.data(), nd, nb * 4, cudaMemcpyDeviceToHost, s->stream));
      SCK(s, cudaMemcpyAsync(den.data(), nd + s->max_batch, nb * 4, cudaMemcpyDeviceToHost, s->stream));
      SCK(s, cudaStreamSynchronize(s->stream));
      for (int q = 0; q < nb; q++)
        sens[b0 + q] = std::max(sens[b0 + q], den[q] > 0.f ? std::sqrt(num[q] / den[q]) : INFINITY);
    }
  }
  return tc_status(s);
}

extern "C" int sur_loss_grad(sur_t *s, const float *X, const float *Y, int n, float *loss, float *grad, size_t ng) {
  if (!s || !X || !Y || n < 1 || n > s->max_batch) return s ? sfail(s, SIM_EINVAL, "bad arguments") : SIM_EINVAL;
  if (grad && ng < (size_t)s->nparam) return sfail(s, SIM_EINVAL, "gradient buffer too small");
  const sur_cfg_t &c = s->cfg;
  const int Lf = L_out(s);
  SCK(s, cudaMemcpyAsync(s->xb, X, (size_t)n * c.in_dim * 4, cudaMemcpyHostToDevice, s->stream));
  SCK(s, cudaMemcpyAsync(s->tb, Y, (size_t)n * Lf * c.out_ch * 4, cudaMemcpyHostToDevice, s->stream));
  SCK(s, forward(s, n));
  SCK(s, backward(s, n, s->lossp));
  std::vector<float> lp(LOSS_PARTS);
  SCK(s, cudaMemcpyAsync(lp.data(), s->lossp, LOSS_PARTS * 4, cudaMemcpyDeviceToHost, s->stream));
  // the gradient kernels run on the handle's (non-blocking) stream: copy on it and wait
  if (grad) SCK(s, cudaMemcpyAsync(grad, s->g, s->nparam * 4, cudaMemcpyDeviceToHost, s->stream));
  SCK(s, cudaStreamSynchronize(s->stream));
  if (loss) *loss = loss_of(s, lp.data(), n);
  return tc_status(s);
}

extern "C" int sur_train(sur_t *s, const float *X, const float *Y, int n, int epochs, int batch, float lr,
                         unsigned long long seed, float *epoch_loss) {
  if (!s || !X || !Y || n < 1 || epochs < 0 || batch < 1 || batch > s->max_batch || !(lr > 0))
    return s ? sfail(s, SIM_EINVAL, "bad training arguments") : SIM_EINVAL;
  SCK(s, cudaSetDevice(s->device));
  const sur_cfg_t &c = s->cfg;
  const int Lf = L_out(s);
  const long long xrow = c.in_dim, yrow = (long long)Lf * c.out_ch;
  const int per_epoch = (n + batch - 1) / batch;
  // the data, the epoch's order and the loss partials of up to LOSS_KEEP
  // minibatches stay on the device, so that no minibatch waits for the host: the
  // losses are read once per epoch, or every LOSS_KEEP minibatches of a longer
  // one (small batches of small cases must not take more memory than their data)
  float *dX = nullptr, *dY = nullptr, *dL = nullptr;
  int *dI = nullptr;
  cudaError_t e = cudaMalloc(&dX, (size_t)n * xrow * 4);
  if (e == cudaSuccess) e = cudaMalloc(&dY, (size_t)n * yrow * 4);
  const int keep = std::min(per_epoch, LOSS_KEEP);
  if (e == cudaSuccess) e = cudaMalloc(&dL, (size_t)keep * LOSS_PARTS * 4);
  if (e == cudaSuccess) e = cudaMalloc(&dI, (size_t)n * 4);
  if (e != cudaSuccess) {
    cudaFree(dX);
    cudaFree(dY);
    cudaFree(dL);
    return sfail(s, SIM_ENOMEM, cudaGetErrorString(e));
  }
  std::vector<float> lp((size_t)keep * LOSS_PARTS);
  e = cudaMemcpyAsync(dX, X, (size_t)n * xrow * 4, cudaMemcpyHostToDevice, s->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(dY, Y, (size_t)n * yrow * 4, cudaMemcpyHostToDevice, s->stream);
  std::vector<int> perm(n);
  for (int q = 0; q < n; q++) perm[q] = q;
  uint64_t st = seed;
  auto rnd = [&]() {
    uint64_t z = (st += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
  };
  const long long steps_total = (long long)epochs * ((n + batch - 1) / batch);
  long long step = 0;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  for (int ep = 0; ep < epochs && e == cudaSuccess; ep++) {
    for (int q = n - 1; q > 0; q--) std::swap(perm[q], perm[rnd() % (uint64_t)(q + 1)]);
    if ((e = cudaMemcpyAsync(dI, perm.data(), (size_t)n * 4, cudaMemcpyHostToDevice, s->stream)) != cudaSuccess) break;
    double lsum = 0;
    int read = 0;  // minibatches whose losses are in lsum
    // the wait also keeps the host's order from being reshuffled before it is uploaded
    auto read_losses = [&](int upto) {
      e = cudaMemcpyAsync(lp.data(), dL, (size_t)(upto - read) * LOSS_PARTS * 4, cudaMemcpyDeviceToHost, s->stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
      for (int q = read; q < upto && e == cudaSuccess; q++)
        lsum += loss_of(s, lp.data() + (size_t)(q - read) * LOSS_PARTS, std::min(batch, n - q * batch));
      read = upto;
    };
    for (int b0 = 0; b0 < n && e == cudaSuccess; b0 += batch) {
      const int nb = std::min(batch, n - b0);
      k_gather<<<egrid(nb * xrow), 256, 0, s->stream>>>(dX, dI + b0, nb, xrow, s->xb);
      k_gather<<<egrid(nb * yrow), 256, 0, s->stream>>>(dY, dI + b0, nb, yrow, s->tb);
      if ((e = forward(s, nb)) != cudaSuccess) break;
      if ((e = backward(s, nb, dL + (size_t)(b0 / batch - read) * LOSS_PARTS)) != cudaSuccess) break;
      // cosine learning-rate schedule over all steps
      const float lr_t = 0.5f * lr * (1.f + cosf(3.14159265f * (float)step / (float)std::max<long long>(1, steps_total)));
      s->adam_t++;
      step++;
      const float c1 = 1.f - powf(b1, (float)s->adam_t), c2 = 1.f - powf(b2, (float)s->adam_t);
      k_adam<<<egrid(s->nparam), 256, 0, s->stream>>>(s->w, s->g, s->m, s->v, s->w16, s->nparam, lr_t, b1, b2, eps, c1,
                                                       c2);
      e = cudaGetLastError();
      const int done = b0 / batch + 1;
      if (e == cudaSuccess && (done - read == keep || done == per_epoch)) read_losses(done);
    }
    if (epoch_loss) epoch_loss[ep] = (float)(lsum / per_epoch);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  cudaFree(dX);
  cudaFree(dY);
  cudaFree(dL);
  cudaFree(dI);
  if (e != cudaSuccess) return sfail(s, SIM_ECUDA, cudaGetErrorString(e));
  return tc_status(s);
}

// fallback gate: errors of validation cases indexed by their normalised inputs
extern "C" int sur_gate_fit(sur_t *s, const float *X, const float *err, int n) {
  if (!s || n < 1 || !X || !err) return s ? sfail(s, SIM_EINVAL, "bad gate data") : SIM_EINVAL;
  const int d = s->cfg.in_dim;
  std::vector<float> mean(d), scale(d);
  SCK(s, cudaStreamSynchronize(s->stream));
  SCK(s, cudaMemcpy(mean.data(), s->x_mean, d * 4, cudaMemcpyDeviceToHost));
  SCK(s, cudaMemcpy(scale.data(), s->x_scale, d * 4, cudaMemcpyDeviceToHost));
  s->gate_x.resize((size_t)n * d);
  s->gate_err.assign(err, err + n);
  for (int q = 0; q < n; q++)
    for (int c = 0; c < d; c++) s->gate_x[(size_t)q * d + c] = (X[(size_t)q * d + c] - mean[c]) / scale[c];
  return SIM_OK;
}

// accept[q] = 1 when the largest error among the k validation cases nearest
// to input q (normalised Euclidean distance) is <= tol
extern "C" int sur_gate(sur_t *s, const float *X, int n, int k, float tol, int *accept) {
  if (!s || n < 0 || (n > 0 && (!X || !accept)) || k < 1) return s ? sfail(s, SIM_EINVAL, "bad gate query") : SIM_EINVAL;
  if (s->gate_err.empty()) return sfail(s, SIM_EINVAL, "gate not fitted");
  const int d = s->cfg.in_dim, m = (int)s->gate_err.size();
  std::vector<float> mean(d), scale(d);
  SCK(s, cudaMemcpy(mean.data(), s->x_mean, d * 4, cudaMemcpyDeviceToHost));
  SCK(s, cudaMemcpy(scale.data(), s->x_scale, d * 4, cudaMemcpyDeviceToHost));
  std::vector<std::pair<float, float>> dist(m);
  for (int q = 0; q < n; q++) {
    for (int j = 0; j < m; j++) {
      float acc = 0;
      for (int c = 0; c < d; c++) {
        const float u = (X[(size_t)q * d + c] - mean[c]) / scale[c] - s->gate_x[(size_t)j * d + c];
        acc += u * u;
      }
      dist[j] = {acc, s->gate_err[j]};
    }
    const int kk = std::min(k, m);
    std::partial_sort(dist.begin(), dist.begin() + kk, dist.end());
    float worst = 0;
    for (int j = 0; j < kk; j++) worst = std::max(worst, dist[j].second);
    accept[q] = worst <= tol ? 1 : 0;
  }
  return SIM_OK;
}

extern "C" void sur_destroy(sur_t *s) {
  if (!s) return;
  cudaSetDevice(s->device);
  if (s->stream) cudaStreamSynchronize(s->stream);
  release_side(s);
  for (void *p : s->allocs) cudaFree(p);
  if (s->own_stream) cudaStreamDestroy(s->stream);
  delete s;
}

extern "C" const char *sur_last_error(const sur_t *s) { return s ? s->err.c_str() : g_sur_err.c_str(); }

// tensor-core GEMM on host buffers (BF16 bit patterns in, FP32 out)
extern "C" int cw_gemm_bf16(int trans_a, int trans_b, int M, int N, int K, const uint16_t *A, int lda,
                            const uint16_t *B, int ldb, float *C, int ldc) {
  return cw_gemm_bf16_path(0, trans_a, trans_b, M, N, K, A, lda, B, ldb, C, ldc);
}

extern "C" int cw_gemm_bf16_path(int path, int trans_a, int trans_b, int M, int N, int K, const uint16_t *A, int lda,
                                 const uint16_t *B, int ldb, float *C, int ldc) {
  if (path < 0 || path > 2 || M < 0 || N < 0 || K < 0 || !A || !B || !C) return SIM_EINVAL;
  const size_t na = (size_t)(trans_a ? K : M) * lda, nb = (size_t)(trans_b ? N : K) * ldb, nc = (size_t)M * ldc;
  __nv_bfloat16 *dA = nullptr, *dB = nullptr;
  float *dC = nullptr;
  cudaError_t e = cudaMalloc(&dA, std::max<size_t>(na, 1) * 2);
  if (e == cudaSuccess) e = cudaMalloc(&dB, std::max<size_t>(nb, 1) * 2);
  if (e == cudaSuccess) e = cudaMalloc(&dC, std::max<size_t>(nc, 1) * 4);
  if (e == cudaSuccess) e = cudaMemcpy(dA, A, na * 2, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dB, B, nb * 2, cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = gemm_path(path, trans_a != 0, trans_b != 0, M, N, K, dA, lda, dB, ldb, dC, ldc, 0);
  if (e == cudaSuccess) e = cudaMemcpy(C, dC, nc * 4, cudaMemcpyDeviceToHost);
  int st = 0;
  if (e == cudaSuccess) e = gemm_tcgen05_status(&st, 0);
  cudaFree(dA);
  cudaFree(dB);
  cudaFree(dC);
  if (e != cudaSuccess) return SIM_ECUDA;
  return st ? SIM_ETIMEOUT : SIM_OK;
}
