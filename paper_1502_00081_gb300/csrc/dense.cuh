// Batched dense complex algebra of the Dyson step, the transmission and the lead decimation: products
// (dyson.cu routes them), LU factorisation and triangular solves (lu.cu).  Column-major matrices.
#pragma once

#include "rsfd_internal.cuh"

namespace rsfd {

// Where the products of a call run: the sliced tensor-core GEMM (oz_gemm.cu) with its digit workspace in
// the handle, or, for small products, without a handle or without memory, the plain kernels.
struct Gemm {
  Handle* h = nullptr;
  cudaStream_t st = nullptr;
  int* err = nullptr;              // device flag of expired waits
  int wait_cap = 0;                // the handle's solve option
  cudaError_t fail = cudaSuccess;  // first launch error
  void note(cudaError_t e) {
    if (e != cudaSuccess && fail == cudaSuccess) fail = e;
  }
};

// C[b] = sign * op(A[b]) B[b] + (add ? C[b] : 0); op = N or conjugate transpose (opA = 1).
// Sliced products hold an element to 2^-62 (FP32: 2^-30) of the largest of its row of op(A) or column of B, not of its own
// size.  ksplit > 0: the sum over k is taken in the ranges [0, ksplit) and [ksplit, k), each with largest elements of its own
// (opA = 0).  The Dyson step needs that at the boundary between the slabs: a column of G has the left slab's part of order 1
// and the right slab's part as small as the transmission amplitude.
void gemm(Gemm& g, int batch, int m, int n, int k, double sign, const double2* A, int lda, long long sA, int opA,
          const double2* B, int ldb, long long sB, bool add, double2* C, int ldc, long long sC, int ksplit = 0);
// the same on the tensor cores, C may be B (without ksplit); false (nothing done) where gemm() would not slice
bool gemm_sliced(Gemm& g, int batch, int m, int n, int k, double sign, const double2* A, int lda, long long sA, int opA,
                 const double2* B, int ldb, long long sB, bool add, double2* C, int ldc, long long sC, int ksplit = 0);
constexpr double kSliceMin = 8e6;   // complex multiply-adds of an FP64 product from which it is sliced
void gemm(Gemm& g, int batch, int m, int n, int k, double sign, const float2* A, int lda, long long sA, int opA,
          const float2* B, int ldb, long long sB, bool add, float2* C, int ldc, long long sC);

constexpr int kSwapInts = 64;   // one panel's row exchanges: 32 destinations, 32 sources
int lu_swap_ints(int nb);       // scratch per matrix of lu_factor, ints

// K matrices nb x nb in place: P M = L U with partial pivoting.  perm [K][nb]: row i of P M is row perm[i] of M;
// info [K] (zeroed by the caller): first column without a usable pivot, 1-based; swp [K][lu_swap_ints(nb)] scratch.
void lu_factor(Gemm& g, double2* M, int nb, int K, int* perm, int* info, int* swp);
void lu_factor(Gemm& g, float2* M, int nb, int K, int* perm, int* info, int* swp);
// inverses of the factors' diagonal blocks for lu_solve with nrhs columns (handle workspace 10, valid until the next
// call), or null where substitution is as fast.  split (0: none): no block of this and of lu_solve holds rows on both sides of
// row split, for the reason given at gemm(); the same value for both.
const double2* lu_inverses(Gemm& g, const double2* LU, int nb, int K, int nrhs, int split);
// X[b] = U^{-1} L^{-1} X[b] for nrhs columns of nb rows (batch stride nb nrhs), rows already permuted
void lu_solve(Gemm& g, const double2* LU, int nb, int K, double2* X, int nrhs, const double2* dinv, int split);
void lu_solve(Gemm& g, const float2* LU, int nb, int K, float2* X, int nrhs, int split);
// X[b][:, c][i] = B[b][:, c][perm[b][i]], with conversion where the types differ; X may be B (same type)
void lu_permute(Gemm& g, const double2* B, int nb, int K, const int* perm, double2* X, int nrhs);
void lu_permute(Gemm& g, const double2* B, int nb, int K, const int* perm, float2* X, int nrhs);

}  // namespace rsfd
