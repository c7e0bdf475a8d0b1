// A batched complex FP32 GEMM on the 5th-generation tensor cores (tcgen05, kind::tf32) with the 3xTF32 split:
// the entry rsfd_cgemm_tf32x3, and the FP32 products of the Dyson step when there is no memory for digit planes.
//
// 3xTF32: every FP32 operand x is split into hi = x with the 13 low mantissa bits cleared (exactly a
// TF32 number) and lo = x - hi (exact in FP32).  A product a*b is taken as
// a_hi*b_hi + a_hi*b_lo + a_lo*b_hi with FP32 accumulation in tensor memory; the dropped a_lo*b_lo
// and the TF32 rounding of lo are ~2^-21 relative, so the GEMM carries FP32-class accuracy.
// Complex C = A B takes four real products: Re = Ar Br - Ai Bi, Im = Ar Bi + Ai Br; the minus sign
// is the instruction descriptor's negate-A bit.  So one K-step of 8 issues 12 MMAs of 128 x BN x 8.
//
// Data path: column-major complex (interleaved re/im) operands are read from global memory by all
// 128 threads, split, and stored into eight shared-memory planes (re_hi, re_lo, im_hi, im_lo of A
// and of B) in the K-major, no-swizzle core-matrix layout of the tensor core (8 rows x 16 bytes per
// core matrix); thread 0 issues the MMAs for a stage and commits them to that stage's mbarrier, so
// the loads of stage s+1 overlap the MMAs of stage s.  The two accumulators (Re, Im: 128 lanes x BN
// FP32 columns each) live in tensor memory and are read back by tcgen05.ld for the epilogue
// C = alpha (Re + i Im) + beta C.

#include <cuda_runtime.h>
#include <stdint.h>

#include "rsfd_internal.cuh"

namespace rsfd {
namespace {

constexpr int TC_BM = 128;        // rows of C per CTA (MMA M)
constexpr int TC_BN = 128;        // columns of C per CTA (MMA N)
constexpr int TC_KC = 16;         // complex K elements per shared-memory stage (two MMA K-steps)
constexpr int TC_THREADS = 128;
constexpr int TC_PLANE_A = TC_BM * TC_KC * 4;   // bytes of one operand plane (8 KB)
constexpr int TC_PLANE_B = TC_BN * TC_KC * 4;
constexpr int TC_STAGE = 4 * TC_PLANE_A + 4 * TC_PLANE_B;
constexpr int TC_NSTAGE = 3;
constexpr int TC_SMEM = TC_NSTAGE * TC_STAGE + 1024;
constexpr int TC_TMEM_COLS = 2 * TC_BN;         // Re and Im accumulators
// core-matrix strides of a plane: 8-row groups are adjacent (128 B apart, the "stride" offset
// along M/N); groups of 4 K-elements are one plane-height apart (the "leading" offset along K)
constexpr uint32_t TC_SBO = 128;
constexpr uint32_t TC_LBO_A = (TC_BM / 8) * 128;
constexpr uint32_t TC_LBO_B = (TC_BN / 8) * 128;
constexpr long long kTcWaitCap = 1ll << 22;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: K-major, no swizzle
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;   // descriptor version of the 5th-generation tensor core
  return d;                 // base offset 0, absolute LBO mode off, layout SWIZZLE_NONE
}

// instruction descriptor of kind::tf32: FP32 accumulator, TF32 A and B, both K-major
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N, int negA) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)negA << 13) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
  for (long long i = 0; i < kTcWaitCap; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void split3(float x, float& hi, float& lo) {
  hi = __uint_as_float(__float_as_uint(x) & 0xFFFFE000u);
  lo = x - hi;
}

// byte offset of element (row, k) inside one plane of `rows` rows (K-major core matrices)
__device__ __forceinline__ uint32_t plane_off(int row, int kgrp, int rows) {
  return (uint32_t)((kgrp * (rows / 8) + (row >> 3)) * 128 + (row & 7) * 16);
}

// C[b] = alpha * A[b] * B[b] + beta * C[b]   (A m x k, B k x n, C m x n, column-major complex FP32)
__global__ void __launch_bounds__(TC_THREADS, 1)
cgemm_tf32x3_kernel(int m, int n, int k, float2 alpha, const float2* __restrict__ A, int lda, long long sA,
                    const float2* __restrict__ B, int ldb, long long sB, float beta, float2* C, int ldc,
                    long long sC, int* err, int vecB) {
  extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
  __shared__ __align__(8) uint64_t bars[TC_NSTAGE];
  __shared__ uint32_t tmem_base_s;
  unsigned char* smem = (unsigned char*)(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int bz = blockIdx.z;
  A += bz * sA;
  B += bz * sB;
  C += bz * sC;
  const int m0 = blockIdx.y * TC_BM, n0 = blockIdx.x * TC_BN;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base_s)),
                 "r"(TC_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int s = 0; s < TC_NSTAGE; ++s)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&bars[s])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base_s;
  const uint32_t tm_re = tmem, tm_im = tmem + TC_BN;

  const int nchunks = (k + TC_KC - 1) / TC_KC;
  const uint32_t id_pos = idesc_tf32(TC_BM, TC_BN, 0), id_neg = idesc_tf32(TC_BM, TC_BN, 1);
  // raw operands of one K-chunk, loaded into registers one chunk ahead of the shared-memory stores:
  // thread tid holds row m0 + tid of A and column n0 + tid of B
  float2 ra[TC_KC], rb[TC_KC];
  auto load_chunk = [&](int kc) {
    const int k0 = kc * TC_KC;
    const int gi = m0 + tid, gj = n0 + tid;
#pragma unroll
    for (int q = 0; q < TC_KC; ++q) {
      const int kk = k0 + q;
      ra[q] = (gi < m && kk < k) ? A[(long long)kk * lda + gi] : make_float2(0.f, 0.f);
    }
    if (vecB && gj < n && k0 + TC_KC <= k) {
      const float4* src = reinterpret_cast<const float4*>(B + (long long)gj * ldb + k0);
#pragma unroll
      for (int q = 0; q < TC_KC / 2; ++q) {
        const float4 v = src[q];
        rb[2 * q] = make_float2(v.x, v.y);
        rb[2 * q + 1] = make_float2(v.z, v.w);
      }
    } else {
#pragma unroll
      for (int q = 0; q < TC_KC; ++q) {
        const int kk = k0 + q;
        rb[q] = (gj < n && kk < k) ? B[(long long)gj * ldb + kk] : make_float2(0.f, 0.f);
      }
    }
  };
  // split into TF32 hi / lo planes in the core-matrix layout of stage st
  auto store_chunk = [&](unsigned char* st) {
    unsigned char* sb = st + 4 * TC_PLANE_A;
#pragma unroll
    for (int g = 0; g < TC_KC / 4; ++g) {
      float rh[4], rl[4], ih[4], il[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        split3(ra[4 * g + q].x, rh[q], rl[q]);
        split3(ra[4 * g + q].y, ih[q], il[q]);
      }
      const uint32_t o = plane_off(tid, g, TC_BM);
      *(float4*)(st + 0 * TC_PLANE_A + o) = make_float4(rh[0], rh[1], rh[2], rh[3]);
      *(float4*)(st + 1 * TC_PLANE_A + o) = make_float4(rl[0], rl[1], rl[2], rl[3]);
      *(float4*)(st + 2 * TC_PLANE_A + o) = make_float4(ih[0], ih[1], ih[2], ih[3]);
      *(float4*)(st + 3 * TC_PLANE_A + o) = make_float4(il[0], il[1], il[2], il[3]);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        split3(rb[4 * g + q].x, rh[q], rl[q]);
        split3(rb[4 * g + q].y, ih[q], il[q]);
      }
      const uint32_t ob = plane_off(tid, g, TC_BN);
      *(float4*)(sb + 0 * TC_PLANE_B + ob) = make_float4(rh[0], rh[1], rh[2], rh[3]);
      *(float4*)(sb + 1 * TC_PLANE_B + ob) = make_float4(rl[0], rl[1], rl[2], rl[3]);
      *(float4*)(sb + 2 * TC_PLANE_B + ob) = make_float4(ih[0], ih[1], ih[2], ih[3]);
      *(float4*)(sb + 3 * TC_PLANE_B + ob) = make_float4(il[0], il[1], il[2], il[3]);
    }
  };
  bool ok = true;
  if (nchunks > 0) load_chunk(0);
  for (int kc = 0; kc < nchunks && ok; ++kc) {
    const int s = kc % TC_NSTAGE;
    unsigned char* st = smem + s * TC_STAGE;
    // the stage is free once the MMAs of chunk kc - TC_NSTAGE (its previous user) have completed
    if (kc >= TC_NSTAGE) ok = bar_wait(smem_addr(&bars[s]), (uint32_t)(((kc - TC_NSTAGE) / TC_NSTAGE) & 1));
    store_chunk(st);
    if (kc + 1 < nchunks) load_chunk(kc + 1);   // in flight while this chunk's MMAs are issued
    // make the generic-proxy stores visible to the tensor core, then issue from one thread
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    ok = __syncthreads_and(ok) != 0;   // uniform: a CTA whose wait expired stops as a whole
    if (!ok) break;
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t a0 = smem_addr(st), b0 = smem_addr(st + 4 * TC_PLANE_A);
#pragma unroll
      for (int t = 0; t < TC_KC / 8; ++t) {
        const uint32_t ka = (uint32_t)(2 * t) * TC_LBO_A, kb = (uint32_t)(2 * t) * TC_LBO_B;
        const uint64_t arh = sdesc(a0 + 0 * TC_PLANE_A + ka, TC_LBO_A, TC_SBO);
        const uint64_t arl = sdesc(a0 + 1 * TC_PLANE_A + ka, TC_LBO_A, TC_SBO);
        const uint64_t aih = sdesc(a0 + 2 * TC_PLANE_A + ka, TC_LBO_A, TC_SBO);
        const uint64_t ail = sdesc(a0 + 3 * TC_PLANE_A + ka, TC_LBO_A, TC_SBO);
        const uint64_t brh = sdesc(b0 + 0 * TC_PLANE_B + kb, TC_LBO_B, TC_SBO);
        const uint64_t brl = sdesc(b0 + 1 * TC_PLANE_B + kb, TC_LBO_B, TC_SBO);
        const uint64_t bih = sdesc(b0 + 2 * TC_PLANE_B + kb, TC_LBO_B, TC_SBO);
        const uint64_t bil = sdesc(b0 + 3 * TC_PLANE_B + kb, TC_LBO_B, TC_SBO);
        const uint32_t acc0 = (kc > 0 || t > 0) ? 1u : 0u;
        // Re += Ar Br - Ai Bi   (small terms first)
        mma_tf32(tm_re, arl, brh, id_pos, acc0);
        mma_tf32(tm_re, arh, brl, id_pos, 1u);
        mma_tf32(tm_re, ail, bih, id_neg, 1u);
        mma_tf32(tm_re, aih, bil, id_neg, 1u);
        mma_tf32(tm_re, arh, brh, id_pos, 1u);
        mma_tf32(tm_re, aih, bih, id_neg, 1u);
        // Im += Ar Bi + Ai Br
        mma_tf32(tm_im, arl, bih, id_pos, acc0);
        mma_tf32(tm_im, arh, bil, id_pos, 1u);
        mma_tf32(tm_im, ail, brh, id_pos, 1u);
        mma_tf32(tm_im, aih, brl, id_pos, 1u);
        mma_tf32(tm_im, arh, bih, id_pos, 1u);
        mma_tf32(tm_im, aih, brh, id_pos, 1u);
      }
      mma_commit(smem_addr(&bars[s]));
    }
  }
  // the last commit covers every MMA issued before it
  if (ok && nchunks > 0)
    ok = bar_wait(smem_addr(&bars[(nchunks - 1) % TC_NSTAGE]), (uint32_t)(((nchunks - 1) / TC_NSTAGE) & 1));
  ok = __syncthreads_and(ok) != 0;
  if (!ok) {
    if (tid == 0) atomicExch(err, 1);
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (ok && nchunks > 0) {
    const int i = m0 + warp * 32 + lane;
    const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
#pragma unroll 1
    for (int c0 = 0; c0 < TC_BN; c0 += 16) {
      if (n0 + c0 >= n) break;   // uniform across the CTA
      float re[16], im[16];
      tmem_ld16(tm_re + lane_off + c0, re);
      tmem_ld16(tm_im + lane_off + c0, im);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (i < m) {
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const int j = n0 + c0 + q;
          if (j < n) {
            float2* c = C + (long long)j * ldc + i;
            float2 out = make_float2(alpha.x * re[q] - alpha.y * im[q], alpha.x * im[q] + alpha.y * re[q]);
            if (beta != 0.f) {
              const float2 old = *c;
              out.x += beta * old.x;
              out.y += beta * old.y;
            }
            *c = out;
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS) : "memory");
}

bool g_tc_attr_set[16] = {false};

}  // namespace

cudaError_t cgemm_tf32x3(cudaStream_t st, int batch, int m, int n, int k, float2 alpha, const float2* A, int lda,
                         long long sA, const float2* B, int ldb, long long sB, float beta, float2* C, int ldc,
                         long long sC, int* err) {
  if (batch <= 0 || m <= 0 || n <= 0) return cudaSuccess;
  if (k <= 0) return cudaErrorInvalidValue;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 16 && !g_tc_attr_set[dev]) {
    e = cudaFuncSetAttribute(cgemm_tf32x3_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    if (e != cudaSuccess) return e;
    g_tc_attr_set[dev] = true;
  }
  dim3 grid((n + TC_BN - 1) / TC_BN, (m + TC_BM - 1) / TC_BM, batch);
  // 16-byte loads of B columns when every column start (B + j ldb + k0, k0 a multiple of 16) is aligned
  const int vecB = ((uintptr_t)B % 16 == 0) && (ldb % 2 == 0) && (sB % 2 == 0);
  cgemm_tf32x3_kernel<<<grid, TC_THREADS, TC_SMEM, st>>>(m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC,
                                                         err, vecB);
  return cudaGetLastError();
}

}  // namespace rsfd

// ------------------------------------------------------------------------------------------------
// C ABI: rsfd_cgemm_tf32x3
// ------------------------------------------------------------------------------------------------
namespace {
__device__ int g_cgemm_err;   // bounded-wait flag of rsfd_cgemm_tf32x3 calls
}

extern "C" rsfd_status rsfd_cgemm_tf32x3(int32_t batch, int32_t m, int32_t n, int32_t k, const double* alpha,
                                         const void* A, int32_t lda, int64_t sA, const void* B, int32_t ldb,
                                         int64_t sB, double beta, void* C, int32_t ldc, int64_t sC, void* stream) {
  if (batch < 0 || m < 0 || n < 0 || k < 1 || !alpha || (beta != 0.0 && beta != 1.0)) return RSFD_ERR_ARG;
  if (batch == 0 || m == 0 || n == 0) return RSFD_OK;
  if (!A || !B || !C || lda < m || ldb < k || ldc < m || sA < 0 || sB < 0 || sC < 0) return RSFD_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  int* err = nullptr;
  if (cudaGetSymbolAddress((void**)&err, g_cgemm_err) != cudaSuccess) return RSFD_ERR_CUDA;
  if (cudaMemsetAsync(err, 0, sizeof(int), st) != cudaSuccess) return RSFD_ERR_CUDA;
  const float2 al = make_float2((float)alpha[0], (float)alpha[1]);
  if (rsfd::cgemm_tf32x3(st, batch, m, n, k, al, (const float2*)A, lda, sA, (const float2*)B, ldb, sB, (float)beta,
                         (float2*)C, ldc, sC, err) != cudaSuccess)
    return RSFD_ERR_CUDA;
  int herr = 0;
  if (cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return RSFD_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return RSFD_ERR_CUDA;
  return herr ? RSFD_ERR_TIMEOUT : RSFD_OK;
}
