// Dyson / OBM boundary step and Fisher-Lee transmission.
//
// G0_bb -> G_bb: the exact relation of Eq. sec3-01a restricted to the boundary rows is the
// linear system (I - G0_bb Sigma_bb) G_bb = G0_bb with Sigma_bb = diag(Sigma_L, Sigma_R)
// (equivalent to the block formulas Eqs. sec3-02 ... sec3-06).  Every energy is an independent
// dense complex solve of size nb; the batch is processed with:
//   1. M = I - G0 Sigma           (batched complex GEMM, FP64)
//   2. M = P L U                  (batched blocked right-looking LU with partial pivoting, lu.cu)
//   3. G = U^{-1} L^{-1} P G0     (batched blocked triangular solves, lu.cu)
//   4. FP64 iterative refinement: R = G0 - M G, G += M^{-1} R (twice), reporting ||R||/||G0||.
// T(E) = Tr[Gamma_L G_RL^H Gamma_R G_RL] (Eq. TF) with Gamma = i (Sigma - Sigma^H) is two
// GEMMs and a trace per energy.  All matrices are column-major per energy.

#include <cuda_runtime.h>
#include <math.h>

#include <cmath>
#include <cstdlib>

#include <string>
#include <vector>

#include "dense.cuh"

namespace rsfd {
namespace {

constexpr int GT = 16;   // GEMM tile

// C[b] = alpha * op(A[b]) * B[b] + beta * C[b];  op = N or H (conjugate transpose).
// A: if opA == 0, m x k (lda); if opA == 1, k x m stored, used as its conjugate transpose.
__global__ void zgemm_batched(int m, int n, int k, double2 alpha, const double2* A, int lda, long long sA, int opA,
                              const double2* B, int ldb, long long sB, double2 beta, double2* C, int ldc,
                              long long sC) {
  __shared__ double2 As[GT][GT + 1];
  __shared__ double2 Bs[GT][GT + 1];
  const int bz = blockIdx.z;
  A += bz * sA;
  B += bz * sB;
  C += bz * sC;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int row = blockIdx.y * GT + ty;   // i in C
  const int col = blockIdx.x * GT + tx;   // j in C
  double2 acc = make_double2(0.0, 0.0);
  for (int k0 = 0; k0 < k; k0 += GT) {
    // A tile: rows blockIdx.y*GT + ty, cols k0 + tx
    {
      const int i = blockIdx.y * GT + ty, kk = k0 + tx;
      double2 v = make_double2(0.0, 0.0);
      if (i < m && kk < k) {
        if (opA == 0) v = A[(long long)kk * lda + i];
        else {
          v = A[(long long)i * lda + kk];
          v.y = -v.y;
        }
      }
      As[ty][tx] = v;
    }
    {
      const int kk = k0 + ty, j = blockIdx.x * GT + tx;
      Bs[ty][tx] = (kk < k && j < n) ? B[(long long)j * ldb + kk] : make_double2(0.0, 0.0);
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < GT; ++t) {
      const double2 a = As[ty][t], b = Bs[t][tx];
      acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
      acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
    }
    __syncthreads();
  }
  if (row < m && col < n) {
    double2* c = C + (long long)col * ldc + row;
    double2 old = (beta.x != 0.0 || beta.y != 0.0) ? *c : make_double2(0.0, 0.0);
    *c = cadd(cmul(alpha, acc), cmul(beta, old));
  }
}

void zgemm(cudaStream_t st, int batch, int m, int n, int k, double2 alpha, const double2* A, int lda, long long sA,
           int opA, const double2* B, int ldb, long long sB, double2 beta, double2* C, int ldc, long long sC) {
  dim3 grid((n + GT - 1) / GT, (m + GT - 1) / GT, batch), block(GT, GT);
  zgemm_batched<<<grid, block, 0, st>>>(m, n, k, alpha, A, lda, sA, opA, B, ldb, sB, beta, C, ldc, sC);
}

// the flag lives in the handle's workspace 9; false: products stay on the CUDA cores
rsfd_status gemm_begin(Handle* h, Gemm& g) {
  g.h = h;
  g.st = handle_stream(h);
  void* p = nullptr;
  const rsfd_status s = handle_ensure(h, 9, 256, &p);
  if (s != RSFD_OK) return s;
  g.err = (int*)p;
  g.wait_cap = handle_wait_cap(h);
  g.fail = cudaMemsetAsync(g.err, 0, sizeof(int), g.st);
  return RSFD_OK;
}

// after the last product: waits for the stream and turns a failed launch or an expired wait into a status
rsfd_status gemm_end(Gemm& g, const char* who) {
  int flag = 0;
  cudaError_t e = g.fail != cudaSuccess ? g.fail : cudaMemcpyAsync(&flag, g.err, sizeof(int), cudaMemcpyDeviceToHost, g.st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(g.st);
  if (e != cudaSuccess) return handle_fail(g.h, RSFD_ERR_CUDA, std::string(who) + ": " + cudaGetErrorString(e));
  if (flag) return handle_fail(g.h, RSFD_ERR_TIMEOUT, std::string(who) + ": tensor-core GEMM wait expired");
  return RSFD_OK;
}

// digits of one product: up to 4 GB for a batch, or what one matrix needs
template <typename T> void* oz_work(Gemm& g, int batch, int m, int n, int k, size_t& bytes) {
  const size_t lim = (size_t)4 << 30, per = oz_bytes(m, n, k, sizeof(T) == 16);
  bytes = per * batch < lim ? per * batch : (per > lim ? per : lim);
  void* w = nullptr;
  return handle_ensure(g.h, 8, bytes, &w) == RSFD_OK ? w : nullptr;
}

}  // namespace

// Sliced from 8e6 complex multiply-adds on: its three launches cost about 17 us a product, which the FP64 pipe
// (1.3e11 complex multiply-adds/s) earns back from there.  Two products of ns x ns x ns and the rest of
// rsfd_transmission, CUDA cores / sliced, us: ns = 64, 16 energies (4.2e6) 143 / 154; 192, 1 (7.1e6) 251 / 266;
// 128, 4 (8.4e6) 242 / 208; 96, 16 (1.4e7) 291 / 190; 256, 16 (2.7e8) 3869 / 600.
bool gemm_sliced(Gemm& g, int batch, int m, int n, int k, double sign, const double2* A, int lda, long long sA, int opA,
                 const double2* B, int ldb, long long sB, bool add, double2* C, int ldc, long long sC, int ksplit) {
  size_t wb = 0;
  const int k1 = ksplit > 0 && ksplit < k ? ksplit : k, k2 = k - k1;
  void* w = g.h && k >= 32 && m >= 32 && n >= 16 && (double)m * n * k * batch >= kSliceMin
                ? oz_work<double2>(g, batch, m, n, k1 > k2 ? k1 : k2, wb)
                : nullptr;
  if (!w) return false;
  const int sg = sign < 0 ? -1 : 1;
  g.note(oz_gemm(g.st, batch, m, n, k1, sg, A, lda, sA, opA, B, ldb, sB, add ? 1 : 0, C, ldc, sC, w, wb, g.err,
                 g.wait_cap));
  if (k2 > 0)
    g.note(oz_gemm(g.st, batch, m, n, k2, sg, A + (long long)k1 * lda, lda, sA, opA, B + k1, ldb, sB, 1, C, ldc, sC, w, wb, g.err,
                 g.wait_cap));
  return true;
}
void gemm(Gemm& g, int batch, int m, int n, int k, double sign, const double2* A, int lda, long long sA, int opA,
          const double2* B, int ldb, long long sB, bool add, double2* C, int ldc, long long sC, int ksplit) {
  if (!gemm_sliced(g, batch, m, n, k, sign, A, lda, sA, opA, B, ldb, sB, add, C, ldc, sC, ksplit))
    zgemm(g.st, batch, m, n, k, make_double2(sign, 0.0), A, lda, sA, opA, B, ldb, sB, make_double2(add ? 1.0 : 0.0, 0.0),
          C, ldc, sC);
}

// FP32 operands (the updates of the FP32 LU and solves): always sliced; without memory for the digits the
// 3xTF32 GEMM.
void gemm(Gemm& g, int batch, int m, int n, int k, double sign, const float2* A, int lda, long long sA, int opA,
          const float2* B, int ldb, long long sB, bool add, float2* C, int ldc, long long sC) {
  size_t wb = 0;
  void* w = oz_work<float2>(g, batch, m, n, k, wb);
  if (w)
    g.note(oz_gemm(g.st, batch, m, n, k, sign < 0 ? -1 : 1, A, lda, sA, opA, B, ldb, sB, add ? 1 : 0, C, ldc, sC, w, wb, g.err,
                 g.wait_cap));
  else
    g.note(cgemm_tf32x3(g.st, batch, m, n, k, make_float2((float)sign, 0.f), A, lda, sA, B, ldb, sB, add ? 1.f : 0.f, C, ldc,
                        sC, g.err));
}

namespace {

template <typename T>
__global__ void to_c128(const T* src, double2* dst, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = make_double2((double)src[i].x, (double)src[i].y);
}
__global__ void from_c128_f(const double2* src, float2* dst, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = make_float2((float)src[i].x, (float)src[i].y);
}
__global__ void copy_c128(const double2* src, double2* dst, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = src[i];
}
__device__ __forceinline__ void cvt(double2 a, double2& b) { b = a; }
__device__ __forceinline__ void cvt(double2 a, float2& b) { b = make_float2((float)a.x, (float)a.y); }
// dst[b ds + i] = src[b ss + i] for i < n, b < batch (a block of leading columns of each energy's
// matrix, with a type conversion where the types differ)
template <typename S, typename D>
__global__ void copy_batched(const S* src, long long ss, D* dst, long long ds, long long n, int batch) {
  const long long tot = n * batch;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot; t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / n, i = t - b * n;
    cvt(src[b * ss + i], dst[b * ds + i]);
  }
}
// dst[b ds + off + i] = 0 for i < n, b < batch
template <typename D>
__global__ void zero_batched(D* dst, long long ds, long long off, long long n, int batch) {
  const long long tot = n * batch;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot; t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / n, i = t - b * n;
    D z;
    z.x = 0;
    z.y = 0;
    dst[b * ds + off + i] = z;
  }
}

// M = I - G0 * blockdiag(SL, SR) is formed by two GEMMs after M = I.
__global__ void set_identity(double2* M, int nb, int batch) {
  const long long n2 = (long long)nb * nb;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n2 * batch;
       t += (long long)gridDim.x * blockDim.x) {
    const long long e = t % n2;
    const long long c = e / nb, r = e - c * nb;
    M[t] = make_double2(r == c ? 1.0 : 0.0, 0.0);
  }
}

__global__ void axpy_c128(double2* y, const double2* x, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = cadd(y[i], x[i]);
}

// Sums over a matrix per batch entry in two launches: kRed blocks an entry leave partial sums in part
// [batch][kRed] (fixed ranges), one warp an entry adds them in order.
constexpr int kRed = 64;
__device__ __forceinline__ double block_sum256(double s) {
  __shared__ double red[8];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < 8; ++w) t += red[w];
  return t;   // thread 0
}
__global__ void __launch_bounds__(256) frob2_part(const double2* A, long long n2, double* part) {
  const double2* a = A + blockIdx.y * n2;
  const long long i1 = n2 * (blockIdx.x + 1) / kRed;
  double s = 0.0;
  for (long long i = n2 * blockIdx.x / kRed + threadIdx.x; i < i1; i += 256) s += cabs2(a[i]);
  s = block_sum256(s);
  if (threadIdx.x == 0) part[blockIdx.y * kRed + blockIdx.x] = s;
}
__global__ void sum_parts(const double* part, double* out, int batch) {
  const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (b >= batch) return;
  double s = 0.0;
  for (int k = lane; k < kRed; k += 32) s += part[b * kRed + k];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) out[b] = s;
}
// the same in one launch without scratch, a block per entry
__global__ void __launch_bounds__(256) frob2_one(const double2* A, long long n2, double* out) {
  const double2* a = A + blockIdx.x * n2;
  double s = 0.0;
  for (long long i = threadIdx.x; i < n2; i += 256) s += cabs2(a[i]);
  s = block_sum256(s);
  if (threadIdx.x == 0) out[blockIdx.x] = s;
}
void frob2_batched(cudaStream_t st, const double2* A, long long n2, int batch, double* part, double* out) {
  frob2_part<<<dim3(kRed, batch), 256, 0, st>>>(A, n2, part);
  sum_parts<<<(batch + 7) / 8, 256, 0, st>>>(part, out, batch);
}

// Gamma = i (S - S^H) for a batch of ns x ns matrices
__global__ void gamma_batched(const double2* S, double2* G, int ns, int batch) {
  const long long n2 = (long long)ns * ns;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n2 * batch;
       t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / n2, e = t - b * n2;
    const int c = (int)(e / ns), r = (int)(e - (long long)c * ns);
    const double2 a = S[t], bt = S[b * n2 + (long long)r * ns + c];   // S[c, r]
    // S - S^H at (r, c) = a - conj(S[c, r]);  times i
    const double2 d = make_double2(a.x - bt.x, a.y + bt.y);
    G[t] = make_double2(-d.y, d.x);
  }
}

// part sums of T[b] = Re sum_{a,c} GL[a,c] W[c,a]: block x of an entry takes a band of 16 x 16 tiles, W through
// shared memory so that both operands are read along their columns
__global__ void __launch_bounds__(256) trace_prod_part(const double2* GL, const double2* W, int ns, double* part) {
  __shared__ double2 tw[16][17];
  const long long n2 = (long long)ns * ns;
  const double2* g = GL + blockIdx.y * n2;
  const double2* w = W + blockIdx.y * n2;
  const int nt = (ns + 15) / 16, tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double s = 0.0;
  for (int t = blockIdx.x; t < nt * nt; t += kRed) {
    const int a0 = (t % nt) * 16, c0 = (t / nt) * 16;
    __syncthreads();
    // W[c, a] sits at a ns + c: read along c
    tw[ty][tx] = (a0 + ty < ns && c0 + tx < ns) ? w[(long long)(a0 + ty) * ns + c0 + tx] : make_double2(0.0, 0.0);
    __syncthreads();
    if (a0 + tx < ns && c0 + ty < ns) {
      const double2 x = g[(long long)(c0 + ty) * ns + a0 + tx], y = tw[tx][ty];
      s += x.x * y.x - x.y * y.y;
    }
  }
  s = block_sum256(s);
  if (threadIdx.x == 0) part[blockIdx.y * kRed + blockIdx.x] = s;
}

// dst[b][c][0:nrow] = src[b][c][0:nrow] for ncol columns: the leading rows of a column-major block
__global__ void copy_rows_c128(const double2* src, int lds, double2* dst, int ldd, int nrow, int ncol, int batch) {
  const long long per = (long long)nrow * ncol;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < per * batch;
       t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / per, e = t - b * per;
    const long long c = e / nrow, i = e - c * nrow;
    dst[(b * ncol + c) * ldd + i] = src[(b * ncol + c) * lds + i];
  }
}

int grid_for(long long n) {
  long long g = (n + 255) / 256;
  return (int)(g < 4096 ? (g < 1 ? 1 : g) : 4096);
}

}  // namespace

#define DY_CK(h, call)                                                                                  \
  do {                                                                                                  \
    cudaError_t e_ = (call);                                                                            \
    if (e_ != cudaSuccess) return handle_fail((h), RSFD_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

__global__ void to_f32_c(const double2* src, float2* dst, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = make_float2((float)src[i].x, (float)src[i].y);
}
__global__ void add_f32_to_c128(double2* y, const float2* x, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = make_double2(y[i].x + (double)x[i].x, y[i].y + (double)x[i].y);
}
__global__ void set_f32_to_c128(double2* y, const float2* x, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = make_double2((double)x[i].x, (double)x[i].y);
}

// Tensor-core form of the Dyson step, energies processed in chunks that fit the device:
//   M = I - G0 Sigma                       FP64 (sliced products)
//   F = P L U of M in FP32                 panels on the CUDA cores, trailing updates sliced (tcgen05)
//   X = F^{-1} G0                          blocked triangular solves, updates sliced (tcgen05)
//   nref times: R = G0 - M X (FP64, sliced), X += F^{-1} R
// Reported residual ||G0 - M X|| / ||G0|| is the FP64 one after the last correction.
rsfd_status dyson_tc_run(Handle* h, const void* G0, const void* SL, const void* SR, int K, void* G, double* refres) {
  const int nb = handle_nb(h);
  const int ns = nb / 2;
  const long long n2 = (long long)nb * nb, s2 = (long long)ns * ns;
  const bool fp64in = handle_prec(h) != RSFD_MIXED;
  const int nref = handle_dyson_refine(h);
  // columns solved: all nb, or the left slab's ns (the block of G_bb the transmission uses)
  const int nc = handle_dyson_cols(h) == 1 ? ns : nb;
  const long long sx = (long long)nb * nc;
  // per energy: M (c128), X, R and the compact right-hand side (c128, nb x nc), the G0 copy when the
  // input is complex64, F (c64) and the FP32 solve (c64, nb x nc)
  const long long per = n2 * (16 + (fp64in ? 0 : 16) + 8) + sx * (3 * 16 + 8) + (long long)nb * 8 + 64;
  size_t free_b = 0, tot_b = 0;
  DY_CK(h, cudaMemGetInfo(&free_b, &tot_b));
  long long kc = (long long)(0.6 * (double)free_b) / per;
  if (kc > K) kc = K;
  if (kc < 1) kc = 1;
  const int Kc = (int)kc;
  rsfd_status s;
  void *pM, *pX, *pR, *pF, *pPiv, *pRed, *pG0, *pB;
  if ((s = handle_ensure(h, 1, n2 * Kc * sizeof(double2), &pM)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 3, sx * Kc * sizeof(double2), &pX)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 4, sx * Kc * sizeof(double2), &pR)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 2, (n2 + sx) * Kc * sizeof(float2), &pF)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 5, (long long)Kc * (nb + 1 + lu_swap_ints(nb)) * sizeof(int), &pPiv)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 6, (long long)(2 + kRed) * K * sizeof(double), &pRed)) != RSFD_OK) return s;
  if (!fp64in && (s = handle_ensure(h, 0, n2 * Kc * sizeof(double2), &pG0)) != RSFD_OK) return s;
  if (nc < nb && (s = handle_ensure(h, 7, sx * Kc * sizeof(double2), &pB)) != RSFD_OK) return s;
  if ((s = handle_begin(h)) != RSFD_OK) return s;
  cudaStream_t st = handle_stream(h);
  Gemm gc;
  if ((s = gemm_begin(h, gc)) != RSFD_OK) return s;
  double2* dM = (double2*)pM;
  double2* dX = (double2*)pX;
  double2* dR = (double2*)pR;
  float2* dF = (float2*)pF;
  float2* dXf = dF + n2 * Kc;
  int* perm = (int*)pPiv;
  int* info = perm + (long long)Kc * nb;
  int* swp = info + Kc;
  double* red = (double*)pRed;
  std::vector<int> hinfo(K, 0);
  for (int k0 = 0; k0 < K; k0 += Kc) {
    const int kb = K - k0 < Kc ? K - k0 : Kc;
    const long long tot = n2 * kb, totx = sx * kb;
    const double2* g0;
    if (fp64in) {
      g0 = (const double2*)G0 + n2 * k0;
    } else {
      to_c128<float2><<<grid_for(tot), 256, 0, st>>>((const float2*)G0 + n2 * k0, (double2*)pG0, tot);
      g0 = (const double2*)pG0;
    }
    // right-hand sides: G0's first nc columns of every energy, compact (stride sx)
    const double2* b0 = g0;
    if (nc < nb) {
      copy_batched<double2, double2><<<grid_for(totx), 256, 0, st>>>(g0, n2, (double2*)pB, sx, sx, kb);
      b0 = (const double2*)pB;
    }
    const double2* sl = (const double2*)SL + s2 * k0;
    const double2* sr = (const double2*)SR + s2 * k0;
    set_identity<<<grid_for(tot), 256, 0, st>>>(dM, nb, kb);
    gemm(gc, kb, nb, ns, ns, -1.0, g0, nb, n2, 0, sl, ns, s2, true, dM, nb, n2);
    gemm(gc, kb, nb, ns, ns, -1.0, g0 + (long long)ns * nb, nb, n2, 0, sr, ns, s2, true, dM + (long long)ns * nb, nb, n2);
    to_f32_c<<<grid_for(tot), 256, 0, st>>>(dM, dF, tot);
    DY_CK(h, cudaMemsetAsync(info, 0, kb * sizeof(int), st));
    lu_factor(gc, dF, nb, kb, perm, info, swp);
    lu_permute(gc, b0, nb, kb, perm, dXf, nc);
    lu_solve(gc, dF, nb, kb, dXf, nc, ns);
    set_f32_to_c128<<<grid_for(totx), 256, 0, st>>>(dX, dXf, totx);
    for (int it = 0; it < nref; ++it) {
      copy_c128<<<grid_for(totx), 256, 0, st>>>(b0, dR, totx);
      gemm(gc, kb, nb, nc, nb, -1.0, dM, nb, n2, 0, dX, nb, sx, true, dR, nb, sx, ns);
      lu_permute(gc, dR, nb, kb, perm, dXf, nc);
      lu_solve(gc, dF, nb, kb, dXf, nc, ns);
      add_f32_to_c128<<<grid_for(totx), 256, 0, st>>>(dX, dXf, totx);
    }
    if (refres) {
      copy_c128<<<grid_for(totx), 256, 0, st>>>(b0, dR, totx);
      gemm(gc, kb, nb, nc, nb, -1.0, dM, nb, n2, 0, dX, nb, sx, true, dR, nb, sx, ns);
      frob2_batched(st, dR, sx, kb, red + 2 * K, red + k0);
      frob2_batched(st, b0, sx, kb, red + 2 * K, red + K + k0);
    }
    if (fp64in) {
      copy_batched<double2, double2><<<grid_for(totx), 256, 0, st>>>(dX, sx, (double2*)G + n2 * k0, n2, sx, kb);
      if (nc < nb) zero_batched<double2><<<grid_for(tot - totx), 256, 0, st>>>((double2*)G + n2 * k0, n2, sx, n2 - sx, kb);
    } else {
      copy_batched<double2, float2><<<grid_for(totx), 256, 0, st>>>(dX, sx, (float2*)G + n2 * k0, n2, sx, kb);
      if (nc < nb) zero_batched<float2><<<grid_for(tot - totx), 256, 0, st>>>((float2*)G + n2 * k0, n2, sx, n2 - sx, kb);
    }
    DY_CK(h, cudaGetLastError());
    DY_CK(h, cudaMemcpyAsync(hinfo.data() + k0, info, kb * sizeof(int), cudaMemcpyDeviceToHost, st));
  }
  std::vector<double> hred(2 * K);
  if (refres) DY_CK(h, cudaMemcpyAsync(hred.data(), red, 2 * K * sizeof(double), cudaMemcpyDeviceToHost, st));
  if ((s = gemm_end(gc, "rsfd_dyson_boundary")) != RSFD_OK) return s;
  if ((s = handle_end(h)) != RSFD_OK) return s;
  if (refres)
    for (int k = 0; k < K; ++k) refres[k] = sqrt(hred[k]) / sqrt(hred[K + k] > 0 ? hred[K + k] : 1.0);
  for (int k = 0; k < K; ++k)
    if (hinfo[k] != 0)
      return handle_fail(h, RSFD_ERR_BREAKDOWN, "rsfd_dyson_boundary: singular I - G0 Sigma at energy " + std::to_string(k));
  return RSFD_OK;
}

rsfd_status dyson_run(Handle* h, const void* G0, const void* SL, const void* SR, int K, void* G, double* refres) {
  if (handle_dyson_kind(h) == RSFD_DYSON_TC) return dyson_tc_run(h, G0, SL, SR, K, G, refres);
  const int nb = handle_nb(h);
  const int ns = nb / 2;
  const long long n2 = (long long)nb * nb;
  const bool fp64 = handle_prec(h) != RSFD_MIXED;   // FP64 and double-float handles hold c128 data
  rsfd_status s;
  void *pG0, *pM, *pLU, *pX, *pR, *pPiv, *pRed;
  if ((s = handle_ensure(h, 0, n2 * K * sizeof(double2), &pG0)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 1, n2 * K * sizeof(double2), &pM)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 2, n2 * K * sizeof(double2), &pLU)) != RSFD_OK) return s;
  // columns solved: all nb, or the left slab's ns (the block of G_bb the transmission uses)
  const int nc = handle_dyson_cols(h) == 1 ? ns : nb;
  const long long sx = (long long)nb * nc, totx = sx * K;
  if ((s = handle_ensure(h, 3, sx * K * sizeof(double2), &pX)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 4, sx * K * sizeof(double2), &pR)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 5, (long long)K * (nb + 1 + lu_swap_ints(nb)) * sizeof(int), &pPiv)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 6, (long long)(2 + kRed) * K * sizeof(double), &pRed)) != RSFD_OK) return s;
  if ((s = handle_begin(h)) != RSFD_OK) return s;
  cudaStream_t st = handle_stream(h);
  Gemm gc;
  if ((s = gemm_begin(h, gc)) != RSFD_OK) return s;
  double2* dG0 = (double2*)pG0;
  double2* dM = (double2*)pM;
  double2* dLU = (double2*)pLU;
  double2* dX = (double2*)pX;
  double2* dR = (double2*)pR;
  int* perm = (int*)pPiv;
  int* info = perm + (long long)K * nb;
  int* swp = info + K;
  double* red = (double*)pRed;
  const long long tot = n2 * K;
  if (fp64) copy_c128<<<grid_for(tot), 256, 0, st>>>((const double2*)G0, dG0, tot);
  else to_c128<float2><<<grid_for(tot), 256, 0, st>>>((const float2*)G0, dG0, tot);
  set_identity<<<grid_for(tot), 256, 0, st>>>(dM, nb, K);
  // M[:, :ns] -= G0[:, :ns] SL ;  M[:, ns:] -= G0[:, ns:] SR
  gemm(gc, K, nb, ns, ns, -1.0, dG0, nb, n2, 0, (const double2*)SL, ns, (long long)ns * ns, true, dM, nb, n2);
  gemm(gc, K, nb, ns, ns, -1.0, dG0 + (long long)ns * nb, nb, n2, 0, (const double2*)SR, ns, (long long)ns * ns, true,
        dM + (long long)ns * nb, nb, n2);
  copy_c128<<<grid_for(tot), 256, 0, st>>>(dM, dLU, tot);
  DY_CK(h, cudaMemsetAsync(info, 0, K * sizeof(int), st));
  lu_factor(gc, dLU, nb, K, perm, info, swp);
  const double2* dinv = lu_inverses(gc, dLU, nb, K, nc, ns);
  // right-hand sides: the first nc columns of every energy, compact (stride sx)
  const double2* b0 = dG0;
  if (nc < nb) {
    void* pB = nullptr;
    if ((s = handle_ensure(h, 7, sx * K * sizeof(double2), &pB)) != RSFD_OK) return s;
    copy_batched<double2, double2><<<grid_for(totx), 256, 0, st>>>(dG0, n2, (double2*)pB, sx, sx, K);
    b0 = (const double2*)pB;
  }
  lu_permute(gc, b0, nb, K, perm, dX, nc);
  lu_solve(gc, dLU, nb, K, dX, nc, dinv, ns);
  // iterative refinement in FP64
  for (int it = 0; it < 2; ++it) {
    copy_c128<<<grid_for(totx), 256, 0, st>>>(b0, dR, totx);
    gemm(gc, K, nb, nc, nb, -1.0, dM, nb, n2, 0, dX, nb, sx, true, dR, nb, sx, ns);
    lu_permute(gc, dR, nb, K, perm, dR, nc);
    lu_solve(gc, dLU, nb, K, dR, nc, dinv, ns);
    axpy_c128<<<grid_for(totx), 256, 0, st>>>(dX, dR, totx);
  }
  if (refres) {
    copy_c128<<<grid_for(totx), 256, 0, st>>>(b0, dR, totx);
    gemm(gc, K, nb, nc, nb, -1.0, dM, nb, n2, 0, dX, nb, sx, true, dR, nb, sx, ns);
    frob2_batched(st, dR, sx, K, red + 2 * K, red);
    frob2_batched(st, b0, sx, K, red + 2 * K, red + K);
  }
  if (fp64) {
    copy_batched<double2, double2><<<grid_for(totx), 256, 0, st>>>(dX, sx, (double2*)G, n2, sx, K);
    if (nc < nb) zero_batched<double2><<<grid_for(tot - totx), 256, 0, st>>>((double2*)G, n2, sx, n2 - sx, K);
  } else {
    copy_batched<double2, float2><<<grid_for(totx), 256, 0, st>>>(dX, sx, (float2*)G, n2, sx, K);
    if (nc < nb) zero_batched<float2><<<grid_for(tot - totx), 256, 0, st>>>((float2*)G, n2, sx, n2 - sx, K);
  }
  DY_CK(h, cudaGetLastError());
  std::vector<int> hinfo(K);
  DY_CK(h, cudaMemcpyAsync(hinfo.data(), info, K * sizeof(int), cudaMemcpyDeviceToHost, st));
  std::vector<double> hred(2 * K);
  if (refres) DY_CK(h, cudaMemcpyAsync(hred.data(), red, 2 * K * sizeof(double), cudaMemcpyDeviceToHost, st));
  if ((s = gemm_end(gc, "rsfd_dyson_boundary")) != RSFD_OK) return s;
  if ((s = handle_end(h)) != RSFD_OK) return s;
  if (refres)
    for (int k = 0; k < K; ++k) refres[k] = sqrt(hred[k]) / sqrt(hred[K + k] > 0 ? hred[K + k] : 1.0);
  for (int k = 0; k < K; ++k)
    if (hinfo[k] != 0)
      return handle_fail(h, RSFD_ERR_BREAKDOWN, "rsfd_dyson_boundary: singular I - G0 Sigma at energy " + std::to_string(k));
  return RSFD_OK;
}

// Dyson step on the recorded rows: G = G0 + G0[:, b] Sigma Y with Y = (I - G0_bb Sigma)^{-1} G0[b, :]
// (the boundary rows of G), all nr x nr per energy, column-major.
rsfd_status dyson_tracked_run(Handle* h, int nr, const void* G0, const void* SL, const void* SR, int K, void* G,
                              double* refres) {
  const int nb = handle_nb(h);
  const int ns = nb / 2;
  const long long r2 = (long long)nr * nr, b2 = (long long)nb * nb, bn = (long long)nb * nr;
  const bool fp64 = handle_prec(h) != RSFD_MIXED;
  rsfd_status s;
  void *pG0, *pM, *pLU, *pY, *pR, *pPiv, *pRed, *pW;
  if ((s = handle_ensure(h, 0, r2 * K * sizeof(double2), &pG0)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 1, b2 * K * sizeof(double2), &pM)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 2, b2 * K * sizeof(double2), &pLU)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 3, bn * K * sizeof(double2), &pY)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 4, bn * K * sizeof(double2), &pR)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 5, (long long)K * (nb + 1 + lu_swap_ints(nb)) * sizeof(int), &pPiv)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 6, (long long)(2 + kRed) * K * sizeof(double), &pRed)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 7, (2 * bn + r2) * K * sizeof(double2), &pW)) != RSFD_OK) return s;
  if ((s = handle_begin(h)) != RSFD_OK) return s;
  cudaStream_t st = handle_stream(h);
  Gemm gc;
  if ((s = gemm_begin(h, gc)) != RSFD_OK) return s;
  double2* dG0 = (double2*)pG0;
  double2* dM = (double2*)pM;
  double2* dLU = (double2*)pLU;
  double2* dY = (double2*)pY;
  double2* dR = (double2*)pR;
  double2* dRHS = (double2*)pW;
  double2* dW = dRHS + bn * K;
  double2* dX = dW + bn * K;
  int* perm = (int*)pPiv;
  int* info = perm + (long long)K * nb;
  int* swp = info + K;
  double* red = (double*)pRed;
  const long long rtot = r2 * K, btot = b2 * K, ntot = bn * K;
  if (fp64) copy_c128<<<grid_for(rtot), 256, 0, st>>>((const double2*)G0, dG0, rtot);
  else to_c128<float2><<<grid_for(rtot), 256, 0, st>>>((const float2*)G0, dG0, rtot);
  // M = I - G0_bb Sigma (G0_bb: the leading nb x nb block of G0, leading dimension nr)
  set_identity<<<grid_for(btot), 256, 0, st>>>(dM, nb, K);
  gemm(gc, K, nb, ns, ns, -1.0, dG0, nr, r2, 0, (const double2*)SL, ns, (long long)ns * ns, true, dM, nb, b2);
  gemm(gc, K, nb, ns, ns, -1.0, dG0 + (long long)ns * nr, nr, r2, 0, (const double2*)SR, ns, (long long)ns * ns, true,
        dM + (long long)ns * nb, nb, b2);
  copy_c128<<<grid_for(btot), 256, 0, st>>>(dM, dLU, btot);
  DY_CK(h, cudaMemsetAsync(info, 0, K * sizeof(int), st));
  lu_factor(gc, dLU, nb, K, perm, info, swp);
  // Y = M^{-1} G0[b, :] with two FP64 refinement steps
  copy_rows_c128<<<grid_for(ntot), 256, 0, st>>>(dG0, nr, dRHS, nb, nb, nr, K);
  const double2* dinv = lu_inverses(gc, dLU, nb, K, nr, ns);
  lu_permute(gc, dRHS, nb, K, perm, dY, nr);
  lu_solve(gc, dLU, nb, K, dY, nr, dinv, ns);
  for (int it = 0; it < 2; ++it) {
    copy_c128<<<grid_for(ntot), 256, 0, st>>>(dRHS, dR, ntot);
    gemm(gc, K, nb, nr, nb, -1.0, dM, nb, b2, 0, dY, nb, bn, true, dR, nb, bn, ns);
    lu_permute(gc, dR, nb, K, perm, dR, nr);
    lu_solve(gc, dLU, nb, K, dR, nr, dinv, ns);
    axpy_c128<<<grid_for(ntot), 256, 0, st>>>(dY, dR, ntot);
  }
  if (refres) {
    copy_c128<<<grid_for(ntot), 256, 0, st>>>(dRHS, dR, ntot);
    gemm(gc, K, nb, nr, nb, -1.0, dM, nb, b2, 0, dY, nb, bn, true, dR, nb, bn, ns);
    frob2_batched(st, dR, bn, K, red + 2 * K, red);
    frob2_batched(st, dRHS, bn, K, red + 2 * K, red + K);
  }
  // W = Sigma Y (block-diagonal Sigma), then G = G0 + G0[:, b] W
  gemm(gc, K, ns, nr, ns, 1.0, (const double2*)SL, ns, (long long)ns * ns, 0, dY, nb, bn, false, dW, nb, bn);
  gemm(gc, K, ns, nr, ns, 1.0, (const double2*)SR, ns, (long long)ns * ns, 0, dY + ns, nb, bn, false, dW + ns, nb, bn);
  copy_c128<<<grid_for(rtot), 256, 0, st>>>(dG0, dX, rtot);
  gemm(gc, K, nr, nr, nb, 1.0, dG0, nr, r2, 0, dW, nb, bn, true, dX, nr, r2, ns);
  if (fp64) copy_c128<<<grid_for(rtot), 256, 0, st>>>(dX, (double2*)G, rtot);
  else from_c128_f<<<grid_for(rtot), 256, 0, st>>>(dX, (float2*)G, rtot);
  DY_CK(h, cudaGetLastError());
  std::vector<int> hinfo(K);
  DY_CK(h, cudaMemcpyAsync(hinfo.data(), info, K * sizeof(int), cudaMemcpyDeviceToHost, st));
  std::vector<double> hred(2 * K);
  if (refres) DY_CK(h, cudaMemcpyAsync(hred.data(), red, 2 * K * sizeof(double), cudaMemcpyDeviceToHost, st));
  if ((s = gemm_end(gc, "rsfd_dyson_tracked")) != RSFD_OK) return s;
  if ((s = handle_end(h)) != RSFD_OK) return s;
  if (refres)
    for (int k = 0; k < K; ++k) refres[k] = sqrt(hred[k]) / sqrt(hred[K + k] > 0 ? hred[K + k] : 1.0);
  for (int k = 0; k < K; ++k)
    if (hinfo[k] != 0)
      return handle_fail(h, RSFD_ERR_BREAKDOWN, "rsfd_dyson_tracked: singular I - G0 Sigma at energy " + std::to_string(k));
  return RSFD_OK;
}

// ------------------------------------------------------------------------------------------------
// Lead self-energies by decimation (Eq. self-energy with the surface Green's function of Eq. surface
// green's function), for leads that repeat one principal layer of R planes with its own potential.
// Principal-layer blocks: H00 (in-plane kinetic + z couplings inside the layer + V), H01 (layer j to
// j+1).  The right lead runs to +z (alpha_0 = H01, beta_0 = H01^T), the left lead to -z (alpha_0 =
// H01^T, beta_0 = H01).  Lopez Sancho-Rubio iteration, batched over energies, all in FP64:
//   g = (Z - eps)^{-1};  eps_s += alpha g beta;  eps += alpha g beta + beta g alpha;
//   alpha = alpha g alpha;  beta = beta g beta;
// until max |alpha|, |beta| fall below 1e-15 max |H01| for every energy; then g_s = (Z - eps_s)^{-1} and
// Sigma_R = H01 g_s H01^T, Sigma_L = H01^T g_s H01.
// ------------------------------------------------------------------------------------------------
__global__ void zi_minus(double2* A, const double2* E, const double2* Z, int n, int batch, int nz) {
  const long long n2 = (long long)n * n;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n2 * batch;
       t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / n2, e = t - b * n2;
    const long long c = e / n, r = e - c * n;
    const double2 v = E[t], z = Z[b % nz];
    A[t] = r == c ? make_double2(z.x - v.x, z.y - v.y) : make_double2(-v.x, -v.y);
  }
}
// dst[b] = src (one n x n matrix broadcast to the batch)
__global__ void bcast_c128(const double2* src, double2* dst, long long n2, int batch) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n2 * batch;
       t += (long long)gridDim.x * blockDim.x)
    dst[t] = src[t % n2];
}
// One step of the iteration around its product P = [alpha; beta] [g alpha, g beta] (2n x 2n; FIRST: alpha and beta are
// given in rhs and there is no product yet):
//   eps_s += alpha g beta;  eps += alpha g beta + beta g alpha;  alpha = alpha g alpha;  beta = beta g beta,
// the next system's A = Z - eps, its right-hand sides rhs = [alpha | beta], the stacked left factor ab = [alpha; beta], and
// the largest |re| + |im| of the new alpha and beta per matrix in mx (bits of a non-negative double; zero before).
template <bool FIRST>
__global__ void __launch_bounds__(256) decimation_step(const double2* P, double2* eps_s, double2* eps, double2* ab, double2* rhs,
                                                       double2* A, const double2* Z, int n, int nz, unsigned long long* mx) {
  const long long n2 = (long long)n * n;
  const int b = blockIdx.y;
  const double2 z = Z[b % nz];
  const double2* p = P + b * 4 * n2;
  double m = 0.0;
  for (long long e = blockIdx.x * 256ll + threadIdx.x; e < n2; e += gridDim.x * 256ll) {
    const int c = (int)(e / n), r = (int)(e - (long long)c * n);
    double2 al, be, ev = eps[b * n2 + e];
    if (FIRST) {
      al = rhs[b * 2 * n2 + e];
      be = rhs[b * 2 * n2 + n2 + e];
    } else {
      const double2* pc = p + (long long)c * 2 * n;
      const double2* pd = p + (long long)(c + n) * 2 * n;
      al = pc[r];
      be = pd[n + r];
      const double2 agb = pd[r], bga = pc[n + r];
      eps_s[b * n2 + e] = cadd(eps_s[b * n2 + e], agb);
      ev = cadd(cadd(ev, agb), bga);
      eps[b * n2 + e] = ev;
      rhs[b * 2 * n2 + e] = al;
      rhs[b * 2 * n2 + n2 + e] = be;
    }
    ab[b * 2 * n2 + (long long)c * 2 * n + r] = al;
    ab[b * 2 * n2 + (long long)c * 2 * n + n + r] = be;
    A[b * n2 + e] = r == c ? make_double2(z.x - ev.x, z.y - ev.y) : make_double2(-ev.x, -ev.y);
    m = fmax(m, fmax(fabs(al.x) + fabs(al.y), fabs(be.x) + fabs(be.y)));   // NaN is passed over
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(mx + b, (unsigned long long)__double_as_longlong(m));
}

static void layer_blocks(int nx, int ny, double hh, int fd_order, const double* V, std::vector<double2>& H00,
                         std::vector<double2>& H01) {
  const int R = fd_order / 2, nxy = nx * ny, n = R * nxy;
  const double c2[2] = {-2.0, 1.0}, c4[3] = {-2.5, 4.0 / 3.0, -1.0 / 12.0};
  const double* c = fd_order == 2 ? c2 : c4;
  double d[3] = {0, 0, 0};
  for (int k = 0; k <= R; ++k) d[k] = -0.5 * c[k] / (hh * hh);
  H00.assign((size_t)n * n, make_double2(0, 0));
  H01.assign((size_t)n * n, make_double2(0, 0));
  auto at = [&](std::vector<double2>& M, int r, int col) -> double2& { return M[(size_t)col * n + r]; };
  for (int a = 0; a < R; ++a)
    for (int y = 0; y < ny; ++y)
      for (int x = 0; x < nx; ++x) {
        const int i = a * nxy + y * nx + x;
        at(H00, i, i).x += 3.0 * d[0] + (V ? V[i] : 0.0);   // x, y, z diagonal parts and the potential
        for (int k = 1; k <= R; ++k) {
          if (x + k < nx) { at(H00, i, i + k).x += d[k]; at(H00, i + k, i).x += d[k]; }
          if (y + k < ny) { at(H00, i, i + k * nx).x += d[k]; at(H00, i + k * nx, i).x += d[k]; }
        }
        for (int cpl = 0; cpl < R; ++cpl) {
          const int j = cpl * nxy + y * nx + x;
          if (cpl != a && std::abs(a - cpl) <= R) at(H00, i, j).x += d[std::abs(a - cpl)];
          const int dist = R + cpl - a;   // plane a of layer j to plane cpl of layer j + 1
          if (dist <= R) at(H01, i, j).x += d[dist];
        }
      }
}

rsfd_status lead_decimation_run(Handle* h, const double* VL, const double* VR, const double* E, int K, double eta,
                                int maxit, void* SLo, void* SRo, int* iters_out) {
  const int nxy = handle_nx(h) * handle_ny(h);
  const int R = handle_fd_order(h) / 2, n = R * nxy;
  const long long n2 = (long long)n * n;
  std::vector<double2> H00L, H00R, H01;
  layer_blocks(handle_nx(h), handle_ny(h), handle_h(h), handle_fd_order(h), VL, H00L, H01);
  layer_blocks(handle_nx(h), handle_ny(h), handle_h(h), handle_fd_order(h), VR, H00R, H01);
  double hmax = 0.0;
  for (const double2& v : H01) hmax = fmax(hmax, fabs(v.x));
  const double tol = 1e-15 * fmax(1.0, hmax);
  std::vector<double2> H01T((size_t)n2);
  for (int r = 0; r < n; ++r)
    for (int c = 0; c < n; ++c) H01T[(size_t)c * n + r] = H01[(size_t)r * n + c];
  // per matrix (an energy has two, the right and the left lead's): eps_s, eps, [alpha; beta], A (LU), Y and rhs (n x 2n),
  // P (2n x 2n)
  const long long per = n2 * 13 * (long long)sizeof(double2) + (n + 1 + lu_swap_ints(n)) * (long long)sizeof(int) + 64;
  size_t free_b = 0, tot_b = 0;
  DY_CK(h, cudaMemGetInfo(&free_b, &tot_b));
  const long long fit = (long long)(0.5 * (double)free_b) / per;
  const int nl = fit < 2 ? 1 : 2;   // both leads in one batch, or one after the other where memory is short
  long long kc = fit / nl;
  if (kc > K) kc = K;
  if (kc > 32767) kc = 32767;
  if (kc < 1) kc = 1;
  const int Kc = (int)kc, Bc = nl * Kc;
  rsfd_status s;
  void *pW, *pC, *pPiv, *pZ;
  if ((s = handle_ensure(h, 1, (size_t)n2 * 13 * Bc * sizeof(double2), &pW)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 2, (size_t)n2 * 4 * sizeof(double2), &pC)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 5, (size_t)Bc * (n + 1 + lu_swap_ints(n)) * sizeof(int), &pPiv)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 6, (size_t)Kc * sizeof(double2) + (size_t)Bc * sizeof(unsigned long long), &pZ)) != RSFD_OK) return s;
  if ((s = handle_begin(h)) != RSFD_OK) return s;
  cudaStream_t st = handle_stream(h);
  Gemm gc;
  if ((s = gemm_begin(h, gc)) != RSFD_OK) return s;
  double2* W = (double2*)pW;
  double2 *eps_s = W, *eps = W + n2 * Bc, *ab = W + 2 * n2 * Bc, *A = W + 4 * n2 * Bc;
  double2 *Y = W + 5 * n2 * Bc, *rhs = W + 7 * n2 * Bc, *P = W + 9 * n2 * Bc;
  double2 *dH00R = (double2*)pC, *dH00L = dH00R + n2, *dH01 = dH00R + 2 * n2, *dH01T = dH00R + 3 * n2;
  int* perm = (int*)pPiv;
  int* info = perm + (long long)Bc * n;
  int* swp = info + Bc;
  // Solves by substitution: nothing refines them, and explicit inverses of the diagonal blocks show.  Error, geometric means,
  // substitution / inverses: closed form at eta 0.01 to 0.05, 64 rows 2.9e-15 / 3.7e-15, 81 rows 2.9e-15 / 5.0e-15 (LAPACK 2.3e-15,
  // 3.2e-15); layers of 200 rows with random potentials against 80-bit arithmetic 3.4e-15 / 5.7e-15.  16 matrices of 200 rows
  // take 38.9 ms, 38.1 with inverses.
  double2* dZ = (double2*)pZ;
  unsigned long long* dmax = (unsigned long long*)(dZ + Kc);
  DY_CK(h, cudaMemcpyAsync(dH00R, H00R.data(), n2 * sizeof(double2), cudaMemcpyHostToDevice, st));
  DY_CK(h, cudaMemcpyAsync(dH00L, H00L.data(), n2 * sizeof(double2), cudaMemcpyHostToDevice, st));
  DY_CK(h, cudaMemcpyAsync(dH01, H01.data(), n2 * sizeof(double2), cudaMemcpyHostToDevice, st));
  DY_CK(h, cudaMemcpyAsync(dH01T, H01T.data(), n2 * sizeof(double2), cudaMemcpyHostToDevice, st));
  int it_max = 0;
  for (int l0 = 0; l0 < 2; l0 += nl)   // lead 0: right, 1: left
  for (int k0 = 0; k0 < K; k0 += Kc) {
    const int kb = K - k0 < Kc ? K - k0 : Kc, nm = nl * kb;   // matrices q kb .. q kb + kb - 1 are lead l0 + q's
    const long long tot = n2 * kb;
    std::vector<double2> Zh(kb);
    for (int k = 0; k < kb; ++k) Zh[k] = make_double2(E[k0 + k], eta);
    DY_CK(h, cudaMemcpyAsync(dZ, Zh.data(), kb * sizeof(double2), cudaMemcpyHostToDevice, st));
    for (int q = 0; q < nl; ++q) {
      const double2* h0 = l0 + q == 0 ? dH00R : dH00L;
      bcast_c128<<<grid_for(tot), 256, 0, st>>>(h0, eps_s + q * tot, n2, kb);
      bcast_c128<<<grid_for(tot), 256, 0, st>>>(h0, eps + q * tot, n2, kb);
    }
    // rhs = [alpha_0 | beta_0]: right [H01 | H01^T], left [H01^T | H01]
    for (int k = 0; k < nm; ++k) {
      const bool right = l0 + k / kb == 0;
      const double2 *a0 = right ? dH01 : dH01T, *b0 = right ? dH01T : dH01;
      DY_CK(h, cudaMemcpyAsync(rhs + k * 2 * n2, a0, n2 * sizeof(double2), cudaMemcpyDeviceToDevice, st));
      DY_CK(h, cudaMemcpyAsync(rhs + k * 2 * n2 + n2, b0, n2 * sizeof(double2), cudaMemcpyDeviceToDevice, st));
    }
    const dim3 gs((unsigned)((n2 + 511) / 512 < 64 ? (n2 + 511) / 512 : 64), nm);
    DY_CK(h, cudaMemsetAsync(dmax, 0, nm * sizeof(unsigned long long), st));
    decimation_step<true><<<gs, 256, 0, st>>>(nullptr, eps_s, eps, ab, rhs, A, dZ, n, kb, dmax);
    int it = 0;
    for (; it < maxit; ++it) {
      std::vector<double> hm(nm);
      DY_CK(h, cudaMemcpyAsync(hm.data(), dmax, nm * sizeof(double), cudaMemcpyDeviceToHost, st));
      DY_CK(h, cudaStreamSynchronize(st));
      bool done = true;
      for (int k = 0; k < nm; ++k) done &= hm[k] < tol;
      if (done) break;
      // Y = g [alpha | beta] by LU of Z - eps, then P = [alpha; beta] Y
      DY_CK(h, cudaMemsetAsync(info, 0, nm * sizeof(int), st));
      lu_factor(gc, A, n, nm, perm, info, swp);
      lu_permute(gc, rhs, n, nm, perm, Y, 2 * n);
      lu_solve(gc, A, n, nm, Y, 2 * n, nullptr, 0);
      gemm(gc, nm, 2 * n, 2 * n, n, 1.0, ab, 2 * n, 2 * n2, 0, Y, n, 2 * n2, false, P, 2 * n, 4 * n2);
      DY_CK(h, cudaMemsetAsync(dmax, 0, nm * sizeof(unsigned long long), st));
      decimation_step<false><<<gs, 256, 0, st>>>(P, eps_s, eps, ab, rhs, A, dZ, n, kb, dmax);
    }
    it_max = it > it_max ? it : it_max;
    // g_s = (Z - eps_s)^{-1}:  Sigma_R = H01 g_s H01^T, Sigma_L = H01^T g_s H01
    zi_minus<<<grid_for(nl * tot), 256, 0, st>>>(A, eps_s, dZ, n, nm, kb);
    DY_CK(h, cudaMemsetAsync(info, 0, nm * sizeof(int), st));
    lu_factor(gc, A, n, nm, perm, info, swp);
    for (int q = 0; q < nl; ++q) bcast_c128<<<grid_for(tot), 256, 0, st>>>(l0 + q == 0 ? dH01T : dH01, rhs + q * tot, n2, kb);
    lu_permute(gc, rhs, n, nm, perm, Y, n);
    lu_solve(gc, A, n, nm, Y, n, nullptr, 0);
    for (int q = 0; q < nl; ++q) {
      const bool right = l0 + q == 0;
      gemm(gc, kb, n, n, n, 1.0, right ? dH01 : dH01T, n, 0, 0, Y + q * tot, n, n2, false,
           (double2*)(right ? SRo : SLo) + n2 * k0, n, n2);
    }
    std::vector<int> hinfo(nm);
    DY_CK(h, cudaMemcpyAsync(hinfo.data(), info, nm * sizeof(int), cudaMemcpyDeviceToHost, st));
    if ((s = gemm_end(gc, "rsfd_lead_sigma_decimation")) != RSFD_OK) return s;
    for (int k = 0; k < nm; ++k)
      if (hinfo[k] != 0)
        return handle_fail(h, RSFD_ERR_BREAKDOWN, "rsfd_lead_sigma_decimation: singular Z - eps at energy " +
                                                      std::to_string(k0 + k % kb));
    if (it >= maxit)
      return handle_fail(h, RSFD_ERR_NOT_CONVERGED, "rsfd_lead_sigma_decimation: no convergence in maxit steps");
  }
  DY_CK(h, cudaGetLastError());
  if ((s = handle_end(h)) != RSFD_OK) return s;
  if (iters_out) *iters_out = it_max;
  return RSFD_OK;
}

rsfd_status transmission_run(Handle* h, const void* G, const void* SL, const void* SR, int K, double* T) {
  const int nb = handle_nb(h);
  const int ns = nb / 2;
  const long long n2 = (long long)nb * nb, s2 = (long long)ns * ns;
  const bool fp64 = handle_prec(h) != RSFD_MIXED;   // FP64 and double-float handles hold c128 data
  rsfd_status s;
  void *pG, *pGL, *pGR, *pW1, *pW2, *pT;
  if ((s = handle_ensure(h, 0, n2 * K * sizeof(double2), &pG)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 1, s2 * K * sizeof(double2), &pGL)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 2, s2 * K * sizeof(double2), &pGR)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 3, s2 * K * sizeof(double2), &pW1)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 4, s2 * K * sizeof(double2), &pW2)) != RSFD_OK) return s;
  if ((s = handle_ensure(h, 6, (long long)(1 + kRed) * K * sizeof(double), &pT)) != RSFD_OK) return s;
  if ((s = handle_begin(h)) != RSFD_OK) return s;
  cudaStream_t st = handle_stream(h);
  Gemm gc;
  if ((s = gemm_begin(h, gc)) != RSFD_OK) return s;
  double2* dG = (double2*)pG;
  const long long tot = n2 * K;
  if (fp64) copy_c128<<<grid_for(tot), 256, 0, st>>>((const double2*)G, dG, tot);
  else to_c128<float2><<<grid_for(tot), 256, 0, st>>>((const float2*)G, dG, tot);
  gamma_batched<<<grid_for(s2 * K), 256, 0, st>>>((const double2*)SL, (double2*)pGL, ns, K);
  gamma_batched<<<grid_for(s2 * K), 256, 0, st>>>((const double2*)SR, (double2*)pGR, ns, K);
  const double2* GRL = dG + ns;   // rows ns.., cols 0..ns-1, leading dimension nb
  // W1 = Gamma_R G_RL ; W2 = G_RL^H W1
  gemm(gc, K, ns, ns, ns, 1.0, (const double2*)pGR, ns, s2, 0, GRL, nb, n2, false, (double2*)pW1, ns, s2);
  gemm(gc, K, ns, ns, ns, 1.0, GRL, nb, n2, 1, (const double2*)pW1, ns, s2, false, (double2*)pW2, ns, s2);
  double* dT = (double*)pT;
  trace_prod_part<<<dim3(kRed, K), 256, 0, st>>>((const double2*)pGL, (const double2*)pW2, ns, dT + K);
  sum_parts<<<(K + 7) / 8, 256, 0, st>>>(dT + K, dT, K);
  DY_CK(h, cudaGetLastError());
  std::vector<double> hT(K);
  DY_CK(h, cudaMemcpyAsync(hT.data(), dT, K * sizeof(double), cudaMemcpyDeviceToHost, st));
  if ((s = gemm_end(gc, "rsfd_transmission")) != RSFD_OK) return s;
  if ((s = handle_end(h)) != RSFD_OK) return s;
  for (int k = 0; k < K; ++k) T[k] = hT[k];
  return RSFD_OK;
}

}  // namespace rsfd

// ------------------------------------------------------------------------------------------------
// Allocation-free variant of the Dyson step.
//
// Some callers cannot allocate device memory at the point where they need the Dyson step: a
// service or framework that has handed its whole device-memory budget to its own caching allocator
// up front (a cudaMalloc then fails, or would take memory that allocator counts on), or a plug-in
// that a host application forbids to change the device's allocation state.  For them,
// rsfd_dyson_boundary_noalloc keeps its scratch (the matrices I - G0 Sigma and their LU factors,
// the refinement residual, the pivots) in the file-scope device array below, which exists for as
// long as the library is loaded on every GPU that loaded it.  The caller passes the inputs and the
// output; nothing is allocated by the call.
// ------------------------------------------------------------------------------------------------
namespace rsfd {
namespace {

constexpr size_t kNoAllocScratchBytes = (size_t)RSFD_NOALLOC_SCRATCH_BYTES;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

// device address of g_noalloc_scratch, looked up once per device (host code must not use the
// symbol itself: on the host it is only a stand-in)
constexpr int kMaxDevices = 64;
static void* g_scratch_ptr[kMaxDevices] = {nullptr};

// first singular energy: *bad starts at K (none) and takes the smallest k with a zero pivot, so the
// message names the same energy as rsfd_dyson_boundary's
__global__ void noalloc_finish(const int* info, const double* red, int K, int* bad, double* ratio) {
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    if (info[k] != 0) atomicMin(bad, k);
    const double g = red[K + k] > 0 ? red[K + k] : 1.0;
    ratio[k] = sqrt(red[k]) / sqrt(g);
  }
}

__global__ void fill_int(int* p, int v) { *p = v; }

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

// Body of rsfd_dyson_boundary_noalloc (the C entry point in rsfd_api.cu wraps it in the ABI's
// exception guard).
rsfd_status dyson_noalloc_run(int32_t nb, int32_t K, const void* G0_bb, const void* Sigma_L, const void* Sigma_R,
                              void* G_bb, double* refine_residual, void* stream) {
  if (nb < 2 || (nb % 2) != 0 || K < 1 || !G0_bb || !Sigma_L || !Sigma_R || !G_bb || G0_bb == G_bb)
    return handle_fail(nullptr, RSFD_ERR_ARG, "rsfd_dyson_boundary_noalloc: bad arguments");
  // the batched kernels put the energy on gridDim.y / gridDim.z
  if (K > 65535)
    return handle_fail(nullptr, RSFD_ERR_ARG,
                       "rsfd_dyson_boundary_noalloc: K = " + std::to_string(K) + " exceeds the limit of 65535 energies per call");
  const long long n2 = (long long)nb * nb;
  const size_t need = 3 * align256((size_t)n2 * K * sizeof(double2)) + align256((size_t)K * (nb + 1) * sizeof(int)) +
                      align256((size_t)3 * K * sizeof(double)) + align256(sizeof(int));
  if (need > kNoAllocScratchBytes)
    return handle_fail(nullptr, RSFD_ERR_ARG,
                       "rsfd_dyson_boundary_noalloc: 3*nb*nb*K*16 bytes plus pivots exceed the " +
                           std::to_string(kNoAllocScratchBytes) + "-byte static scratch (nb=" + std::to_string(nb) +
                           ", K=" + std::to_string(K) + ")");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return handle_fail(nullptr, RSFD_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return handle_fail(nullptr, RSFD_ERR_ARG, "rsfd_dyson_boundary_noalloc: device index too large");
  if (!g_scratch_ptr[dev]) {   // one-time set-up on this device (the current device)
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
      return handle_fail(nullptr, RSFD_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    g_scratch_ptr[dev] = p;
  }
  unsigned char* base = (unsigned char*)g_scratch_ptr[dev];
  double2* dM = (double2*)base;
  base += align256((size_t)n2 * K * sizeof(double2));
  double2* dLU = (double2*)base;
  base += align256((size_t)n2 * K * sizeof(double2));
  double2* dR = (double2*)base;
  base += align256((size_t)n2 * K * sizeof(double2));
  int* perm = (int*)base;
  int* info = perm + (size_t)K * nb;
  base += align256((size_t)K * (nb + 1) * sizeof(int));
  double* red = (double*)base;   // [2K] squared norms, [K] ratios
  base += align256((size_t)3 * K * sizeof(double));
  int* bad = (int*)base;
  base += align256(sizeof(int));
  // the LU's exchange lists: behind the rest, or, when that is full, in the residual's place (not yet in use,
  // and at least as large from nb = 4 on)
  const size_t swp_bytes = (size_t)K * lu_swap_ints(nb) * sizeof(int);
  int* swp = need + swp_bytes <= kNoAllocScratchBytes ? (int*)base : (int*)dR;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  Gemm gc;   // no handle: the CUDA-core products
  gc.st = st;
  const double2* G0 = (const double2*)G0_bb;
  double2* dX = (double2*)G_bb;
  const long long tot = n2 * K;
  // the scratch keeps the previous call's contents: clear the flags that must start at zero
  e = cudaMemsetAsync(info, 0, K * sizeof(int), st);
  if (e != cudaSuccess) return handle_fail(nullptr, RSFD_ERR_CUDA, std::string("cudaMemsetAsync: ") + cudaGetErrorString(e));
  fill_int<<<1, 1, 0, st>>>(bad, K);
  set_identity<<<grid_for(tot), 256, 0, st>>>(dM, nb, K);
  const int ns = nb / 2;
  gemm(gc, K, nb, ns, ns, -1.0, G0, nb, n2, 0, (const double2*)Sigma_L, ns, (long long)ns * ns, true, dM, nb, n2);
  gemm(gc, K, nb, ns, ns, -1.0, G0 + (long long)ns * nb, nb, n2, 0, (const double2*)Sigma_R, ns, (long long)ns * ns, true,
        dM + (long long)ns * nb, nb, n2);
  copy_c128<<<grid_for(tot), 256, 0, st>>>(dM, dLU, tot);
  lu_factor(gc, dLU, nb, K, perm, info, swp);
  lu_permute(gc, G0, nb, K, perm, dX, nb);
  lu_solve(gc, dLU, nb, K, dX, nb, nullptr, 0);
  for (int it = 0; it < 2; ++it) {
    copy_c128<<<grid_for(tot), 256, 0, st>>>(G0, dR, tot);
    gemm(gc, K, nb, nb, nb, -1.0, dM, nb, n2, 0, dX, nb, n2, true, dR, nb, n2);
    lu_permute(gc, dR, nb, K, perm, dR, nb);
    lu_solve(gc, dLU, nb, K, dR, nb, nullptr, 0);
    axpy_c128<<<grid_for(tot), 256, 0, st>>>(dX, dR, tot);
  }
  copy_c128<<<grid_for(tot), 256, 0, st>>>(G0, dR, tot);
  gemm(gc, K, nb, nb, nb, -1.0, dM, nb, n2, 0, dX, nb, n2, true, dR, nb, n2);
  frob2_one<<<K, 256, 0, st>>>(dR, n2, red);
  frob2_one<<<K, 256, 0, st>>>(G0, n2, red + K);
  noalloc_finish<<<1, 256, 0, st>>>(info, red, K, bad, red + 2 * K);
  e = gc.fail != cudaSuccess ? gc.fail : cudaGetLastError();
  int hbad = K;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && refine_residual)
    e = cudaMemcpyAsync(refine_residual, red + 2 * K, K * sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return handle_fail(nullptr, RSFD_ERR_CUDA, std::string("rsfd_dyson_boundary_noalloc: ") + cudaGetErrorString(e));
  if (hbad < K)
    return handle_fail(nullptr, RSFD_ERR_BREAKDOWN,
                       "rsfd_dyson_boundary_noalloc: singular I - G0 Sigma at energy " + std::to_string(hbad));
  return RSFD_OK;
}

}  // namespace rsfd
