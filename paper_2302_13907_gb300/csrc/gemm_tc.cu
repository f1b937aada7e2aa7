// BF16 GEMM on the fifth-generation tensor cores (tcgen05, accumulator in
// tensor memory) for the trace surrogate.
//
//   C[M x N] = op(A)[M x K] * op(B)[K x N]
//
// A and B are BF16 row-major (op = transpose when TA / TB), C FP32 row-major.
// One CTA of four warps computes a 128 x NT tile of C, NT = 128 or, for
// narrower products, N rounded up to 16:
//  * warp 0 allocates the TMEM columns of the FP32 accumulator (TMEM lane m =
//    tile row m, column n = tile column n);
//  * per K chunk of 64 the four warps stage op(A) rows and op(B) columns in
//    shared memory in the no-swizzle K-major core-matrix layout (8 rows x 16
//    bytes per core matrix; core matrices 128 bytes apart along K, 1024 bytes
//    apart along M / N), zero-filling the ragged edges;
//  * one thread issues four tcgen05.mma (K = 16 each) and commits them to an
//    mbarrier; with more than one chunk the next one is staged into a second
//    buffer meanwhile, and a buffer is waited for (bounded) before it is refilled;
//  * the epilogue reads the accumulator with tcgen05.ld (warp w reads TMEM
//    lanes 32 w .. 32 w + 31, 16 columns per load) and writes C.
// A wait that gives up sets bit 0 of the GEMM status word and skips the
// epilogue; the block then waits (bounded) once more for the MMAs it
// committed, and the TMEM columns are always freed.
//
// The surrogate's products are at most 67 MFLOP: what bounds them is one
// CTA's latency (load, MMA, read back) and the reads and writes of A and C.
// So the operands come in as 16-byte loads, all of a thread's eight issued
// before the first is stored, whichever index of the source is contiguous
// (the earlier element-wise staging of a [K][N] operand, 64 dependent 2-byte
// loads per thread, was most of a 23 us kernel), and a narrow product takes
// only the shared memory and TMEM columns its NT needs, so that more CTAs
// share an SM.
#include "cwell_internal.cuh"
#include "tma_util.cuh"

namespace cwell {
namespace {

constexpr int TBM = 128, TBN = 128, TBK = 64;
constexpr int A_ELEMS = TBM * TBK;  // 128 x 64 BF16 = 16 KB

__device__ int g_tc_status;

// shared-memory matrix descriptor: start address, leading (K-direction) and
// stride (M/N-direction) byte offsets between core matrices, descriptor
// version 1, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// instruction descriptor, kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N = nt, M = TBM
__device__ __forceinline__ uint32_t instr_desc(int nt) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(nt >> 3) << 17) | ((uint32_t)(TBM >> 4) << 24);
}

// the first min(n, 8) BF16 values at src, zero-filled to 8, as one 16-byte word
__device__ __forceinline__ uint4 pack8(const __nv_bfloat16 *src, int n) {
  uint32_t w[4];
#pragma unroll
  for (int e = 0; e < 4; e++) {
    const uint32_t lo = 2 * e < n ? __bfloat16_as_ushort(src[2 * e]) : 0u;
    const uint32_t hi = 2 * e + 1 < n ? __bfloat16_as_ushort(src[2 * e + 1]) : 0u;
    w[e] = lo | (hi << 16);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// element (row, k) of a staged tile in the core-matrix layout
__device__ __forceinline__ int cm_off(int row, int k) {
  return ((row >> 3) * (TBK / 8) + (k >> 3)) * 64 + (row & 7) * 8 + (k & 7);
}

// Stage rows r0 .. r0 + rows - 1 (rows a multiple of 16, those from R on zero)
// and columns k0 .. k0 + 63 (from K on zero) of an operand.  KC: K is the
// contiguous index of the source, element (r, k) at src[r ld + k]; a 16-byte
// word is one row of a core matrix, eight lanes fill a core matrix (no bank
// conflict) and a warp reads 64 contiguous bytes of eight rows.  Otherwise
// element (r, k) at src[k ld + r]: a 16-byte word is eight rows of one k,
// stored as eight 2-byte values.  vec: the source's rows are 16-byte aligned.
template <bool KC>
__device__ __forceinline__ void stage_op(__nv_bfloat16 *dst, const __nv_bfloat16 *__restrict__ src, int ld, int r0, int R,
                                         int rows, int k0, int K, bool vec) {
  const int G = rows >> 3, total = G * TBK;  // 16-byte words
  for (int q0 = threadIdx.x; q0 < total; q0 += 128 * 8) {
    uint4 v[8];
    int at[8];
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int q = q0 + 128 * u, t = q >> 3;
      const int r = KC ? (q & 7) + (t >> 3) * 8 : (t % G) * 8, k = KC ? (t & 7) * 8 : (q & 7) + (t / G) * 8;
      at[u] = q < total ? cm_off(r, k) : -1;
      v[u] = make_uint4(0u, 0u, 0u, 0u);
      const int gr = r0 + r, gk = k0 + k, n = KC ? (gr < R ? K - gk : 0) : (gk < K ? R - gr : 0);
      if (q < total && n > 0) {
        const __nv_bfloat16 *g = src + (KC ? (long long)gr * ld + gk : (long long)gk * ld + gr);
        v[u] = vec && n >= 8 ? __ldg(reinterpret_cast<const uint4 *>(g)) : pack8(g, n);
      }
    }
#pragma unroll
    for (int u = 0; u < 8; u++)
      if (at[u] >= 0) {
        if (KC) {
          *reinterpret_cast<uint4 *>(dst + at[u]) = v[u];
        } else {
          const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
          for (int e = 0; e < 8; e++)
            dst[at[u] + 8 * e] = __ushort_as_bfloat16((unsigned short)(w[e >> 1] >> (16 * (e & 1))));
        }
      }
  }
}

// nt: tile columns, cols: TMEM columns (a power of two, >= 32 and >= nt), nbuf: staging buffers (1 or 2)
template <bool TA, bool TB>
__global__ void __launch_bounds__(128) gemm_tc(int M, int N, int K, const __nv_bfloat16 *__restrict__ A, int lda,
                                               const __nv_bfloat16 *__restrict__ B, int ldb, float *__restrict__ C,
                                               int ldc, int nt, int cols, int nbuf) {
  extern __shared__ __align__(128) unsigned char smem[];
  __nv_bfloat16 *buf = reinterpret_cast<__nv_bfloat16 *>(smem);
  const int buf_elems = A_ELEMS + nt * TBK;
  __shared__ uint64_t bar[2];
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.y * TBM, n0 = blockIdx.x * nt;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tslot)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tslot;

  const int nk = (K + TBK - 1) / TBK;
  const bool vec_a = (lda % 8) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  const bool vec_b = (ldb % 8) == 0 && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
  const uint32_t idesc = instr_desc(nt);
  bool fail = false;
  int issued = 0;  // chunks whose MMAs have been committed; chunk c is use c / nbuf of bar[c % nbuf]
  for (int kc = 0; kc < nk; kc++) {
    const int b = kc % nbuf;
    __nv_bfloat16 *As = buf + b * buf_elems, *Bs = As + A_ELEMS;
    const bool ok = kc < nbuf || mbar_wait(&bar[b], (kc / nbuf - 1) & 1);  // its last MMAs have read the buffer
    stage_op<!TA>(As, A, lda, m0, M, TBM, kc * TBK, K, vec_a);
    stage_op<TB>(Bs, B, ldb, n0, N, nt, kc * TBK, K, vec_b);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (__syncthreads_or(!ok)) {
      fail = true;
      break;
    }
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int ks = 0; ks < TBK / 16; ks++) {
        const uint64_t ad = smem_desc(smem_u32(As) + ks * 256, 128, 1024);
        const uint64_t bd = smem_desc(smem_u32(Bs) + ks * 256, 128, 1024);
        const uint32_t acc = (kc > 0 || ks > 0) ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
            : "memory");
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                       smem_u32(&bar[b]))
                   : "memory");
    }
    issued = kc + 1;
  }
  if (!fail && nk > 0) fail = __syncthreads_or(!mbar_wait(&bar[(nk - 1) % nbuf], ((nk - 1) / nbuf) & 1));
  // after a give-up the MMAs committed last may still be writing the
  // accumulator: wait (bounded) once more for those commits before the columns
  // are freed, so that a later CTA allocating them finds them quiet
  if (fail)
    for (int c = issued > nbuf ? issued - nbuf : 0; c < issued; c++) (void)mbar_wait(&bar[c % nbuf], (c / nbuf) & 1);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  if (!fail) {
    const int m = m0 + 32 * warp + lane;
    const bool vec_c = (ldc % 4) == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
#pragma unroll 1
    for (int c0 = 0; c0 < nt && n0 + c0 < N; c0 += 16) {
      uint32_t r[16];
      if (nk > 0) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
            "%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      } else {
#pragma unroll
        for (int c = 0; c < 16; c++) r[c] = 0u;  // K = 0: the product is zero
      }
      if (m < M) {
        float *cp = C + (long long)m * ldc + n0 + c0;
#pragma unroll
        for (int c = 0; c < 16; c += 4) {
          if (vec_c && n0 + c0 + c + 4 <= N) {
            *reinterpret_cast<float4 *>(cp + c) = make_float4(__uint_as_float(r[c]), __uint_as_float(r[c + 1]),
                                                              __uint_as_float(r[c + 2]), __uint_as_float(r[c + 3]));
          } else {
#pragma unroll
            for (int e = 0; e < 4; e++)
              if (n0 + c0 + c + e < N) cp[c + e] = __uint_as_float(r[c + e]);
          }
        }
      }
    }
  } else if (tid == 0) {
    atomicOr(&g_tc_status, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}

template <bool TA, bool TB>
cudaError_t launch_tc_t(int M, int N, int K, const __nv_bfloat16 *A, int lda, const __nv_bfloat16 *B, int ldb,
                        float *C, int ldc, cudaStream_t s) {
  const int nt = N >= TBN ? TBN : (N + 15) / 16 * 16;
  const int cols = nt <= 32 ? 32 : nt <= 64 ? 64 : 128;
  const int nbuf = K > TBK ? 2 : 1;
  // shared memory asked per CTA: the staging buffers, and at least the share
  // that keeps the resident CTAs' accumulators within the SM's 512 TMEM columns
  const int need = nbuf * (A_ELEMS + nt * TBK) * 2, share = 56 * 1024 * cols / 128;
  const int bytes = need > share ? need : share;
  cudaError_t e = cudaFuncSetAttribute(gemm_tc<TA, TB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 32 * 1024);
  if (e != cudaSuccess) return e;
  dim3 grd((N + nt - 1) / nt, (M + TBM - 1) / TBM);
  gemm_tc<TA, TB><<<grd, 128, bytes, s>>>(M, N, K, A, lda, B, ldb, C, ldc, nt, cols, nbuf);
  return cudaGetLastError();
}

}  // namespace

cudaError_t gemm_tcgen05(bool ta, bool tb, int M, int N, int K, const __nv_bfloat16 *A, int lda,
                         const __nv_bfloat16 *B, int ldb, float *C, int ldc, cudaStream_t s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (K < 0 || (M + TBM - 1) / TBM > 65535) return cudaErrorInvalidValue;
  if (!ta && !tb) return launch_tc_t<false, false>(M, N, K, A, lda, B, ldb, C, ldc, s);
  if (!ta && tb) return launch_tc_t<false, true>(M, N, K, A, lda, B, ldb, C, ldc, s);
  if (ta && !tb) return launch_tc_t<true, false>(M, N, K, A, lda, B, ldb, C, ldc, s);
  return launch_tc_t<true, true>(M, N, K, A, lda, B, ldb, C, ldc, s);
}

// reads and clears the status word of the tcgen05 GEMM (bit 0: a bounded wait gave up)
cudaError_t gemm_tcgen05_status(int *out, cudaStream_t s) {
  cudaError_t e = cudaMemcpyFromSymbolAsync(out, g_tc_status, sizeof(int), 0, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess && *out) {
    const int z = 0;
    e = cudaMemcpyToSymbolAsync(g_tc_status, &z, sizeof(int), 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  }
  return e;
}

}  // namespace cwell
