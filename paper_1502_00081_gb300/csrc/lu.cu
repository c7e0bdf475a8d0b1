// Batched LU with partial pivoting and triangular solves in FP32 and FP64 complex arithmetic, for the
// boundary solve (I - G0 Sigma) G = G0 (Eq. sec3-01a) and the lead decimation.
//
// Right-looking, two levels.  Outer blocks of 128 (FP32) or 64 (FP64) columns end in one tensor-core product
// A22 -= L21 U12; FP64 takes the narrower block because the updates inside it run on the FP64 pipe.  Inside an outer block,
// panels of W columns take three launches:
//   lu_panel   factorises rows x W: every row of the panel lives in one thread's registers, the rows are
//              spread over up to 8 CTAs of a cluster, and a column costs one block and one cluster barrier
//              (the pivot candidates, the pivot row and the row it replaces travel through
//              distributed shared memory);
//   lu_swap    applies the panel's exchanges to the outer block's other columns as one permutation of at
//              most 2 W rows, and solves with the panel's unit lower triangle for those to its right;
//   lu_update  the rank-W update of the rest of the outer block.
// The exchanges then reach the other columns (lu_swap_rest), and U12 = L11^{-1} A12 is a triangular solve.
// Triangular solves: blocks of 64 (FP64) or 128 (FP32) rows by substitution (lu_trsm), the rest by products.  In the Dyson
// step no block of a solve holds rows of both slabs (dense.cuh); the factorisation's blocks may, there the parts that a product
// loses are squares of the coupling beside elements of order 1.
//
// Measured (16 matrices of 1024 rows, FP32 LU and two solves of 1024 columns): panel_getrf + laswp + trsm + 3xTF32
// updates 48 ms before, 11 ms now; 4 of 2048: 123 -> 17 ms; 8 of 512 in FP64 with three solves of 512 columns: 213 ->
// 8 ms (one thread a column before).  The FP64 panel step: 6.3 us a column with FP64 compares, Smith reciprocals and
// rows fetched after the barrier, 4.2 us as it is.
// What bounds it: the panels are a chain of nb column steps (two barriers, a reciprocal and the row update each); the
// FP64 pipe for lu_update, lu_trsm and lu_invert in FP64; the products run at tensor rate.

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "dense.cuh"

namespace cg = cooperative_groups;

namespace rsfd {
namespace {

constexpr int kPanelThreads = 512;
constexpr int kMaxCluster = 8;   // portable cluster size
constexpr int kMaxPanels = 16;   // panels of an outer block (at least 8 columns each)

template <typename T> struct Num;
template <> struct Num<float2> {
  typedef float R;
  static constexpr int NBLK = 128;   // columns per outer block = k of the products, and rows per substitution block
  // pivot measure, as in the FP32 form's reference: |re| + |im|
  static __device__ __forceinline__ float mag(float2 a) { return fabsf(a.x) + fabsf(a.y); }
  static __device__ __forceinline__ float2 mul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
  }
  // c - a b
  static __device__ __forceinline__ float2 nma(float2 a, float2 b, float2 c) {
    return make_float2(fmaf(-a.x, b.x, fmaf(a.y, b.y, c.x)), fmaf(-a.x, b.y, fmaf(-a.y, b.x, c.y)));
  }
  static __device__ __forceinline__ float2 recip(float2 d) {   // Smith
    if (d.x == 0.f && d.y == 0.f) return make_float2(0.f, 0.f);
    if (fabsf(d.x) >= fabsf(d.y)) {
      const float r = d.y / d.x, den = d.x + d.y * r;
      return make_float2(1.f / den, -r / den);
    }
    const float r = d.x / d.y, den = d.y + d.x * r;
    return make_float2(r / den, -1.f / den);
  }
};
template <> struct Num<double2> {
  typedef double R;
  static constexpr int NBLK = 64;
  static __device__ __forceinline__ double mag(double2 a) { return cabs2(a); }
  static __device__ __forceinline__ double2 mul(double2 a, double2 b) { return cmul(a, b); }
  static __device__ __forceinline__ double2 nma(double2 a, double2 b, double2 c) {
    return make_double2(fma(-a.x, b.x, fma(a.y, b.y, c.x)), fma(-a.x, b.y, fma(-a.y, b.x, c.y)));
  }
  static __device__ __forceinline__ double2 recip(double2 d) {
    if (d.x == 0.0 && d.y == 0.0) return make_double2(0.0, 0.0);
    // d* / |d|^2 with d scaled to a component near 1 (no overflow or underflow): one division instead of Smith's three
    const int hx = __double2hiint(d.x) & 0x7ff00000, hy = __double2hiint(d.y) & 0x7ff00000;
    const int h = hx > hy ? hx : hy;
    if (h < 0x00200000 || h > 0x7fd00000) return cdiv(make_double2(1.0, 0.0), d);   // near the ends of the range
    const double s = __hiloint2double(0x7fe00000 - h, 0);
    const double x = d.x * s, y = d.y * s, q = s / fma(x, x, y * y);
    return make_double2(x * q, -y * q);
  }
};

__device__ __forceinline__ float2 shfl(float2 v, int l) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}
__device__ __forceinline__ double2 shfl(double2 v, int l) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}

// The panel's exchanges (row j0 + t with row piv[t], t = 0 .. jw - 1 in order) as one permutation of at
// most 2 W rows: entry e moves row src[e] to row dst[e] (dst < 0: unused).  One warp.
template <int W> __device__ void swap_list(const int* piv, int j0, int jw, int* out) {
  const int lane = threadIdx.x & 31;
  int row = -1 - lane;
  if (lane < W) {
    if (lane < jw) row = j0 + lane;
  } else if (lane < 2 * W && lane - W < jw) {
    row = piv[lane - W];
  }
  const int first = __ffs(__match_any_sync(0xffffffffu, row)) - 1;   // the entry that stands for this row
  int label = row;
  for (int t = 0; t < jw; ++t) {
    const int q = __shfl_sync(0xffffffffu, first, W + t);
    const int a = __shfl_sync(0xffffffffu, label, t), c = __shfl_sync(0xffffffffu, label, q);
    if (lane == t) label = c;
    if (lane == q) label = a;
  }
  const bool valid = row >= 0 && lane == first;
  out[lane] = valid ? row : -1;
  out[32 + lane] = label;
}

// Pivot keys: the leading word of the pivot measure, ordered like it as an integer (-1 for NaN, 0 only for 0).  The search
// compares FP64 measures to 20 bits, which moves the growth bound by 1e-6 and takes it off the FP64 pipe.
__device__ __forceinline__ int pivot_key(float v) { return v == v ? __float_as_int(v) : -1; }
__device__ __forceinline__ int pivot_key(double v) {
  const int hi = __double2hiint(v);
  return v == v ? (hi == 0 && __double2loint(v) != 0 ? 1 : hi) : -1;
}

// Factorise columns j0 .. j0 + jw - 1 (jw <= W <= 16) of matrix blockIdx.y, rows j0 .. nb - 1; grid (cluster size, K).
// Ties in the pivot search go to the lowest row.  What a column step waits for: two warp reductions, one block
// barrier, the reciprocal of the candidate pivots, one cluster barrier; every CTA pushes its candidate row (and the one
// that holds row j also that row) into the shared memory of all before the barrier, so nothing is fetched after it.
template <typename T, int W, int RPT>
__global__ void __launch_bounds__(kPanelThreads) lu_panel(T* M, int nb, int j0, int jw, int* swp, int ss, int* info) {
  typedef Num<T> N;
  cg::cluster_group cl = cg::this_cluster();
  const int C = gridDim.x, rank = blockIdx.x, b = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nw = nt >> 5;
  // what the CTAs show each other, double-buffered by column parity: a CTA that writes for column jj + 2 has passed
  // the barrier of column jj + 1, at which every CTA has finished reading what belongs to column jj.
  // s_cand[.][r]: candidate row of CTA r and, last, the reciprocal of its pivot
  __shared__ T s_cand[2][kMaxCluster][W + 1], s_rowj[2][W];
  __shared__ int2 s_best[2][kMaxCluster];   // key and row of every CTA's candidate
  __shared__ int2 s_wbest[kPanelThreads / 32];
  __shared__ int s_piv[W];
  T* A = M + (long long)b * nb * nb + (long long)j0 * nb;
  const int row0 = j0 + rank * nt * RPT + tid;
  T a[RPT][W];
#pragma unroll
  for (int r = 0; r < RPT; ++r)
#pragma unroll
    for (int c = 0; c < W; ++c) {
      const int i = row0 + r * nt;
      a[r][c] = (i < nb && c < jw) ? A[(long long)c * nb + i] : T();
    }
  if (C > 1) cl.sync();   // every CTA of the cluster runs before its shared memory is written
  // The current column is always register 0; after a column the registers move down by one, its values to the end.  In
  // FP32 the column loop is not unrolled: 16 copies of it, 60 KB of code that runs once, were bound by instruction fetch
  // (2048 rows: 50 us a panel, 23 us rolled).  In FP64, bound by its pipe, the unrolled loop is the faster one (37.7
  // against 39.7 ms for 13 factorisations and solves of 16 x 200 rows) and the moves are free.
  constexpr int kUnroll = sizeof(T) == 16 ? W : 1;
#pragma unroll kUnroll
  for (int jj = 0; jj < W; ++jj) {
    if (jj < jw) {
      const int gj = j0 + jj, par = jj & 1;
      int key = -1, bi = 0x7fffffff;
#pragma unroll
      for (int r = 0; r < RPT; ++r) {
        const int i = row0 + r * nt;
        const int v = i >= gj && i < nb ? pivot_key(N::mag(a[r][0])) : -1;
        if (v > key) {
          key = v;
          bi = i;
        }
      }
      {
        const int m = __reduce_max_sync(0xffffffffu, key);
        bi = __reduce_min_sync(0xffffffffu, key == m && m >= 0 ? bi : 0x7fffffff);
        if (lane == 0) s_wbest[warp] = make_int2(m, bi);
      }
      if (rank == 0 && warp == 0) {   // row gj, in thread jj's registers, to every CTA
        T* src = &s_rowj[par][0];
        if (tid == jj) {
#pragma unroll
          for (int c = 0; c < W; ++c) src[c] = a[0][c];
        }
        __syncwarp();
        for (int e = lane; e < W * (C - 1); e += 32) cl.map_shared_rank(src, 1 + e / W)[e % W] = src[e % W];
      }
      __syncthreads();
      {
        const int2 w = lane < nw ? s_wbest[lane] : make_int2(-1, 0x7fffffff);
        const int m = __reduce_max_sync(0xffffffffu, w.x);
        key = m;
        bi = __reduce_min_sync(0xffffffffu, w.x == m && m >= 0 ? w.y : 0x7fffffff);
      }
      // the candidate's warp pushes its row; warp 0 pushes key and row number
      bool mine = false;
#pragma unroll
      for (int r = 0; r < RPT; ++r) mine |= row0 + r * nt == bi;
      if (__any_sync(0xffffffffu, mine)) {
        T* src = &s_cand[par][rank][0];
#pragma unroll
        for (int r = 0; r < RPT; ++r)
          if (row0 + r * nt == bi) {
#pragma unroll
            for (int c = 0; c < W; ++c) src[c] = a[r][c];
            src[W] = N::recip(a[r][0]);
          }
        __syncwarp();
        for (int e = lane; e < (W + 1) * (C - 1); e += 32) {
          const int o = e / (W + 1), c = e % (W + 1);
          cl.map_shared_rank(src, o + (o >= rank ? 1 : 0))[c] = src[c];
        }
      }
      if (warp == 0 && lane < C) *cl.map_shared_rank(&s_best[par][rank], lane) = make_int2(key, bi);
      if (C > 1) cl.sync();
      else __syncthreads();
      int pr;
      {
        const int2 w = lane < C ? s_best[par][lane] : make_int2(-1, 0x7fffffff);
        key = __reduce_max_sync(0xffffffffu, w.x);
        bi = __reduce_min_sync(0xffffffffu, w.x == key && key >= 0 ? w.y : 0x7fffffff);
      }
      const bool none = key < 0;   // no comparable entry in the column (all NaN)
      const int gp = none ? gj : bi;
      pr = (gp - j0) / (nt * RPT);
      const T* prow = none ? &s_rowj[par][0] : &s_cand[par][pr][0];
      const T* jrow = &s_rowj[par][0];
      const T inv = none ? T() : s_cand[par][pr][W];
      if (rank == 0 && tid == 0) {
        s_piv[jj] = gp;
        if ((none || key == 0) && info[b] == 0) info[b] = gj + 1;   // no pivot, or one of measure zero
      }
#pragma unroll
      for (int r = 0; r < RPT; ++r) {
        const int i = row0 + r * nt;
        if (gp != gj && (i == gp || i == gj)) {
          const T* o = i == gp ? jrow : prow;
#pragma unroll
          for (int c = 0; c < W; ++c) a[r][c] = o[c];
        }
        if (i > gj && i < nb) {
          const T l = N::mul(a[r][0], inv);
          a[r][0] = l;
#pragma unroll
          for (int c = 1; c < W; ++c)
            if (c < W - jj) a[r][c] = N::nma(l, prow[c], a[r][c]);   // the others are finished columns
        }
      }
    }
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
      const T t = a[r][0];
#pragma unroll
      for (int c = 0; c + 1 < W; ++c) a[r][c] = a[r][c + 1];
      a[r][W - 1] = t;
    }
  }
#pragma unroll
  for (int r = 0; r < RPT; ++r)
#pragma unroll
    for (int c = 0; c < W; ++c) {
      const int i = row0 + r * nt;
      if (i < nb && c < jw) A[(long long)c * nb + i] = a[r][c];
    }
  __syncthreads();
  if (rank == 0 && warp == 0) swap_list<W>(s_piv, j0, jw, swp + (long long)b * ss);
}

// The same for panels taller than the clusters hold: one CTA per matrix, the panel stays in global memory.
template <typename T>
__global__ void __launch_bounds__(kPanelThreads) lu_panel_global(T* M, int nb, int j0, int jw, int* swp, int ss,
                                                               int* info) {
  typedef Num<T> N;
  typedef typename N::R R;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, nt = blockDim.x;
  T* A = M + (long long)b * nb * nb;
  __shared__ R s_wv[kPanelThreads / 32];
  __shared__ int s_wi[kPanelThreads / 32];
  __shared__ T s_inv;
  __shared__ int s_piv[16];
  for (int j = j0; j < j0 + jw; ++j) {
    R best = (R)-1;
    int bi = 0x7fffffff;
    for (int i = j + tid; i < nb; i += nt) {
      const R v = N::mag(A[(long long)j * nb + i]);
      if (v > best) {
        best = v;
        bi = i;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const R ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) {
        best = ov;
        bi = oi;
      }
    }
    if (lane == 0) {
      s_wv[tid >> 5] = best;
      s_wi[tid >> 5] = bi;
    }
    __syncthreads();
    best = s_wv[0];
    bi = s_wi[0];
    for (int w = 1; w < nt >> 5; ++w)
      if (s_wv[w] > best || (s_wv[w] == best && s_wi[w] < bi)) {
        best = s_wv[w];
        bi = s_wi[w];
      }
    const int p = bi == 0x7fffffff ? j : bi;
    if (tid == 0) {
      s_piv[j - j0] = p;
      if (!(best > (R)0) && info[b] == 0) info[b] = j + 1;
    }
    if (p != j && tid < jw) {
      T* c = A + (long long)(j0 + tid) * nb;
      const T t = c[j];
      c[j] = c[p];
      c[p] = t;
    }
    __syncthreads();
    if (tid == 0) s_inv = N::recip(A[(long long)j * nb + j]);
    __syncthreads();
    const T inv = s_inv;
    for (int i = j + 1 + tid; i < nb; i += nt) {
      const T l = N::mul(A[(long long)j * nb + i], inv);
      A[(long long)j * nb + i] = l;
      for (int c = j + 1; c < j0 + jw; ++c) A[(long long)c * nb + i] = N::nma(l, A[(long long)c * nb + j], A[(long long)c * nb + i]);
    }
    __syncthreads();
  }
  if (tid < 32) swap_list<16>(s_piv, j0, jw, swp + (long long)b * ss);
}

// Row exchanges of the panel (W, j0, jw) in the outer block's other columns o0 .. oend - 1, one thread per column;
// those right of the panel are also solved with its unit lower triangle.  Bound: latency of 2 W scattered
// loads per thread, all in flight together, and in FP64 the pipe (so a CTA is one warp).
template <typename T, int W>
__global__ void __launch_bounds__(32) lu_swap(T* M, int nb, int o0, int oend, int j0, int jw, const int* swp, int ss) {
  typedef Num<T> N;
  const int b = blockIdx.y;
  __shared__ int s_dst[2 * W], s_src[2 * W];
  __shared__ T s_L[W][W];
  T* A = M + (long long)b * nb * nb;
  const int* sw = swp + (long long)b * ss;
  for (int t = threadIdx.x; t < 2 * W; t += 32) {
    s_dst[t] = sw[t];
    s_src[t] = sw[32 + t];
  }
#pragma unroll
  for (int i = 0; i < W * W / 32; ++i) {
    const int t = i * 32 + threadIdx.x, c = t / W, r = t % W;
    s_L[r][c] = (r > c && r < jw) ? A[(long long)(j0 + c) * nb + j0 + r] : T();
  }
  __syncthreads();
  const int c = o0 + blockIdx.x * 32 + threadIdx.x;
  if (c >= oend || (c >= j0 && c < j0 + jw)) return;
  T* col = A + (long long)c * nb;
  const bool right = c >= j0 + jw;
  T v[2 * W];
#pragma unroll
  for (int t = 0; t < 2 * W; ++t) {
    v[t] = T();
    if (s_dst[t] >= 0 && (s_dst[t] != s_src[t] || (right && t < W))) v[t] = col[s_src[t]];
  }
  if (right) {
#pragma unroll
    for (int q = 0; q < W - 1; ++q)   // by columns: the updates of one q are independent
#pragma unroll
      for (int r = q + 1; r < W; ++r) v[r] = N::nma(s_L[r][q], v[q], v[r]);
  }
#pragma unroll
  for (int t = 0; t < 2 * W; ++t)
    if (s_dst[t] >= 0 && (s_dst[t] != s_src[t] || (right && t < W))) col[s_dst[t]] = v[t];
}

// The exchanges of an outer block's np panels, in order, in the columns outside it and in perm (the last
// "column"), one thread per column.
template <typename V> __device__ __forceinline__ void apply_lists(V* col, const int (*lists)[kSwapInts], int np) {
  for (int p = 0; p < np; ++p) {
    V v[32];
#pragma unroll
    for (int t = 0; t < 32; ++t)
      if (lists[p][t] >= 0 && lists[p][t] != lists[p][32 + t]) v[t] = col[lists[p][32 + t]];
#pragma unroll
    for (int t = 0; t < 32; ++t)
      if (lists[p][t] >= 0 && lists[p][t] != lists[p][32 + t]) col[lists[p][t]] = v[t];
  }
}
template <typename T>
__global__ void __launch_bounds__(64) lu_swap_rest(T* M, int nb, int o0, int oend, int np, const int* swp, int ss, int* perm) {
  __shared__ int s_l[kMaxPanels][kSwapInts];
  const int b = blockIdx.y;
  for (int t = threadIdx.x; t < np * kSwapInts; t += blockDim.x) s_l[t / kSwapInts][t % kSwapInts] = swp[(long long)b * ss + t];
  __syncthreads();
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= o0) c += oend - o0;
  if (c > nb) return;
  if (c == nb) apply_lists(perm + (long long)b * nb, s_l, np);
  else apply_lists(M + (long long)b * nb * nb + (long long)c * nb, s_l, np);
}

// A[i, c] -= sum_t A[i, j0 + t] A[j0 + t, c] for rows r0 .. nb - 1 of columns r0 .. oend - 1 (r0 = j0 + jw).  Tiles of 64
// rows x 16 columns, 128 threads.
template <typename T, int W>
__global__ void __launch_bounds__(128) lu_update(T* M, int nb, int j0, int jw, int oend) {
  typedef Num<T> N;
  __shared__ T s_u[16][W];
  const int r0 = j0 + jw;
  T* A = M + (long long)blockIdx.z * nb * nb;
  const int rb = r0 + blockIdx.x * 64, cb = r0 + blockIdx.y * 16;
  for (int e = threadIdx.x; e < 16 * W; e += 128) {
    const int c = cb + e / W, q = e % W;
    s_u[e / W][q] = (c < oend && q < jw) ? A[(long long)c * nb + j0 + q] : T();
  }
  __syncthreads();
  const int i = rb + (threadIdx.x & 63), cg0 = (threadIdx.x >> 6) * 8;
  if (i >= nb) return;
  T l[W];
#pragma unroll
  for (int q = 0; q < W; ++q) l[q] = q < jw ? A[(long long)(j0 + q) * nb + i] : T();
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int c = cb + cg0 + e;
    if (c < oend) {
      T v = A[(long long)c * nb + i];
#pragma unroll
      for (int q = 0; q < W; ++q) v = N::nma(l[q], s_u[cg0 + e][q], v);
      A[(long long)c * nb + i] = v;
    }
  }
}

// X[r0 .. r0 + ib, :] = T^{-1} X[r0 .. r0 + ib, :] for the diagonal block T of LU at (r0, r0): unit lower (LOWER) or
// upper triangle.  Eight threads share a column (rows q, q + 8, ...), 32 columns per CTA of 256 threads (4 per
// warp; FP64 takes CTAs of one warp, so that the FP64 pipes of all SMs have their share); T passes through
// shared memory in strips of 16 columns, only as many as the block has rows for (all of them for every block: 0.64 instead of 0.50
// ms for the interior planes of 18 boundary rows, 40.9 instead of 38.9 ms for the decimation of 200 rows, whose last block has 8); the
// solved element travels by shuffle.  X has nb rows and batch stride sX.  Bound: FP64 (FP32) pipe.
// INV: X is the identity and the result goes to D (64 x 64, one of a matrix's diagonal blocks' inverses).
template <typename T, bool LOWER, bool INV>
__device__ __forceinline__ void trsm_body(const T* LU, int nb, int r0, int ib, T* X, long long sX, int nrhs, int b, T* D) {
  typedef Num<T> N;
  constexpr int NB = Num<T>::NBLK, RP = NB / 8, NS = NB / 16;
  __shared__ T s_t[16][NB];
  __shared__ T s_d[NB];
  const int tid = threadIdx.x, lane = tid & 31, q = tid & 7;
  const int nt = blockDim.x, col = blockIdx.x * (nt >> 3) + (tid >> 3);
  const T* F = LU + (long long)b * nb * nb + (long long)r0 * nb + r0;
  T* x = X + b * sX + (long long)col * nb + r0;
  if (!LOWER)
    for (int i = tid; i < ib; i += nt) s_d[i] = N::recip(F[(long long)i * nb + i]);
  T v[RP];
#pragma unroll
  for (int k = 0; k < RP; ++k) {
    const int r = k * 8 + q;
    if (INV) {
      v[k] = T();
      if (r == col) v[k].x = 1;
    } else {
      v[k] = (col < nrhs && r < ib) ? x[r] : T();
    }
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const int i0 = (LOWER ? s : NS - 1 - s) * 16;
    if (i0 >= ib) continue;   // uniform: a short block has no such rows
    __syncthreads();
    for (int e = tid; e < 16 * NB; e += nt) {
      const int c = e / NB, r = e % NB;
      s_t[c][r] = (i0 + c < ib && r < ib) ? F[(long long)(i0 + c) * nb + r] : T();
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int t = LOWER ? u : 15 - u;
      const int ki = (LOWER ? s : NS - 1 - s) * 2 + t / 8;   // register of row i = i0 + t in its owner (q = t % 8)
      T xi = shfl(v[ki], (lane & 24) | (t & 7));
      if (!LOWER) {
        if (i0 + t < ib) {   // uniform
          xi = N::mul(xi, s_d[i0 + t]);
          if (q == (t & 7)) v[ki] = xi;
        }
      }
#pragma unroll
      for (int k = 0; k < RP; ++k) {
        if (LOWER ? k > ki : k < ki) v[k] = N::nma(s_t[t][k * 8 + q], xi, v[k]);
        if (k == ki && (LOWER ? q > (t & 7) : q < (t & 7))) v[k] = N::nma(s_t[t][k * 8 + q], xi, v[k]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < RP; ++k) {
    const int r = k * 8 + q;
    if (INV) D[(long long)col * NB + r] = v[k];
    else if (col < nrhs && r < ib) x[r] = v[k];
  }
}
template <typename T, bool LOWER>
__global__ void __launch_bounds__(256, sizeof(T) == 16 ? 2 : 3) lu_trsm(const T* LU, int nb, int r0, int ib, T* X,
                                                                         long long sX, int nrhs) {
  trsm_body<T, LOWER, false>(LU, nb, r0, ib, X, sX, nrhs, blockIdx.y, nullptr);
}
// Blocks of at most NB rows of [0, n), none of them across row split (0: no such row)
struct RowBlocks {
  int n, NB, split, n1;   // n1 blocks end at split
  __host__ __device__ RowBlocks(int n_, int NB_, int split_)
      : n(n_), NB(NB_), split(split_ < n_ ? split_ : 0), n1((split + NB_ - 1) / NB_) {}
  __host__ __device__ int count() const { return n1 + (n - split + NB - 1) / NB; }
  __host__ __device__ int row(int b) const { return b < n1 ? b * NB : split + (b - n1) * NB; }
  __host__ __device__ int rows(int b) const {
    const int left = (b < n1 ? split : n) - row(b);
    return left < NB ? left : NB;
  }
};

// Inverses of the diagonal blocks of (at most) 64 rows, for solves whose products run on the tensor cores: block (z >> 1) of
// matrix blockIdx.y, its unit lower (z even) or upper (z odd) triangle; dinv [K][blocks][2][64 x 64].  One warp per 4 columns.
__global__ void __launch_bounds__(32) lu_invert(const double2* LU, int nb, int split, double2* dinv) {
  constexpr int NB = Num<double2>::NBLK;
  const RowBlocks bl(nb, NB, split);
  const int blk = blockIdx.z >> 1, r0 = bl.row(blk), ib = bl.rows(blk), nblk = bl.count();
  double2* D = dinv + (((long long)blockIdx.y * nblk + blk) * 2 + (blockIdx.z & 1)) * NB * NB;
  if (blockIdx.z & 1) trsm_body<double2, false, true>(LU, nb, r0, ib, nullptr, 0, NB, blockIdx.y, D);
  else trsm_body<double2, true, true>(LU, nb, r0, ib, nullptr, 0, NB, blockIdx.y, D);
}

__global__ void iota_rows(int* perm, int nb, int K) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < (long long)nb * K;
       t += (long long)gridDim.x * blockDim.x)
    perm[t] = (int)(t % nb);
}

__device__ __forceinline__ void conv(double2 a, double2& r) { r = a; }
__device__ __forceinline__ void conv(double2 a, float2& r) { r = make_float2((float)a.x, (float)a.y); }

// X[:, c][i] = B[:, c][perm[i]] between different buffers
template <typename S, typename T>
__global__ void permute_rows(const S* B, int nb, int nrhs, const int* perm, T* X, int K) {
  const long long per = (long long)nb * nrhs;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < per * K; t += (long long)gridDim.x * blockDim.x) {
    const long long b = t / per, e = t - b * per;
    const long long c = e / nb, i = e - c * nb;
    conv(B[b * per + c * nb + perm[b * nb + i]], X[t]);
  }
}
// in place, one column per CTA through shared memory
__global__ void permute_rows_inplace(double2* X, int nb, int nrhs, const int* perm) {
  extern __shared__ double2 s_col[];
  double2* x = X + ((long long)blockIdx.y * nrhs + blockIdx.x) * nb;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) s_col[i] = x[i];
  __syncthreads();
  const int* pm = perm + (long long)blockIdx.y * nb;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) x[i] = s_col[pm[i]];
}

int grid1(long long n) {
  const long long g = (n + 255) / 256;
  return (int)(g < 8192 ? (g < 1 ? 1 : g) : 8192);
}

template <typename T, int W, int RPT>
void launch_panel(Gemm& g, T* M, int nb, int K, int j0, int jw, int C, int* swp, int ss, int* info) {
  const int rows = nb - j0;
  const int per = (rows + C * RPT - 1) / (C * RPT);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C, K);
  cfg.blockDim = dim3((per + 31) / 32 * 32);
  cfg.stream = g.st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = C;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  g.note(cudaLaunchKernelEx(&cfg, lu_panel<T, W, RPT>, M, nb, j0, jw, swp, ss, info));
}

template <typename T, int W>
void launch_swap_update(Gemm& g, T* M, int nb, int K, int o0, int j0, int jw, int oend, const int* swp, int ss) {
  if (oend - o0 > jw) lu_swap<T, W><<<dim3((oend - o0 + 31) / 32, K), 32, 0, g.st>>>(M, nb, o0, oend, j0, jw, swp, ss);
  const int r0 = j0 + jw;
  if (r0 < oend) lu_update<T, W><<<dim3((nb - r0 + 63) / 64, (oend - r0 + 15) / 16, K), 128, 0, g.st>>>(M, nb, j0, jw, oend);
}

// Panel width and rows per thread by the panel's height: a row takes W registers pairs (quads in FP64), a
// thread holds 64 of them, and a cluster has at most 8 x 512 threads.  FP64 panels are spread over the cluster
// from 64 rows per CTA on (an SM does two FP64 FMAs a clock), FP32 panels from 512.
template <typename T>
int panel(Gemm& g, T* M, int nb, int K, int o0, int j0, int oend, int* info, int* swp, int ss) {
  constexpr bool dbl = sizeof(T) == 16;
  const int rows = nb - j0, left = oend - j0;
  const int top = kMaxCluster * kPanelThreads;
  auto cluster = [&](int per) {
    const int c = (rows + per - 1) / per;
    return c < 1 ? 1 : (c > kMaxCluster ? kMaxCluster : c);
  };
  int jw;
  if (rows <= top) {
    jw = left < 16 ? left : 16;
    launch_panel<T, 16, 1>(g, M, nb, K, j0, jw, cluster(dbl ? 64 : kPanelThreads), swp, ss, info);
    launch_swap_update<T, 16>(g, M, nb, K, o0, j0, jw, oend, swp, ss);
  } else if (rows <= 2 * top) {
    constexpr int W = dbl ? 8 : 16;
    jw = left < W ? left : W;
    launch_panel<T, W, 2>(g, M, nb, K, j0, jw, kMaxCluster, swp, ss, info);
    launch_swap_update<T, W>(g, M, nb, K, o0, j0, jw, oend, swp, ss);
  } else if (!dbl && rows <= 4 * top) {
    jw = left < 8 ? left : 8;
    launch_panel<T, 8, dbl ? 2 : 4>(g, M, nb, K, j0, jw, kMaxCluster, swp, ss, info);
    launch_swap_update<T, 8>(g, M, nb, K, o0, j0, jw, oend, swp, ss);
  } else {
    jw = left < 16 ? left : 16;
    lu_panel_global<T><<<K, kPanelThreads, 0, g.st>>>(M, nb, j0, jw, swp, ss, info);
    launch_swap_update<T, 16>(g, M, nb, K, o0, j0, jw, oend, swp, ss);
  }
  return jw;
}

// X = T^{-1} X for the unit lower triangle (LOWER) or the upper triangle of rows and columns r0 .. r1 - 1 of LU, in blocks
// that do not cross row r0 + split.  dinv: the diagonal blocks' inverses (FP64, r0 = 0), or null for substitution.
template <typename T, bool LOWER>
void solve_range(Gemm& g, const T* LU, int nb, int K, int r0, int r1, T* X, long long sX, int nrhs, const T* dinv, int split) {
  constexpr int NB = Num<T>::NBLK;
  const long long n2 = (long long)nb * nb;
  const int thr = sizeof(T) == 16 ? 32 : 256, per = thr / 8;
  const dim3 grid((nrhs + per - 1) / per, K);
  const RowBlocks bl(r1 - r0, NB, split);
  const int nblk = bl.count();
  for (int bi = 0; bi < nblk; ++bi) {
    const int blk = LOWER ? bi : nblk - 1 - bi, s0 = r0 + bl.row(blk), ib = bl.rows(blk);
    bool done = false;
    if constexpr (sizeof(T) == 16) {
      // X_b = T_bb^{-1} X_b in place: the digits of X_b are taken before the product is written
      if (dinv)
        done = gemm_sliced(g, K, ib, nrhs, ib, 1.0, dinv + ((long long)blk * 2 + (LOWER ? 0 : 1)) * NB * NB, NB,
                           (long long)nblk * 2 * NB * NB, 0, X + s0, nb, sX, false, X + s0, nb, sX);
    }
    if (!done) lu_trsm<T, LOWER><<<grid, thr, 0, g.st>>>(LU, nb, s0, ib, X, sX, nrhs);
    const int d0 = LOWER ? s0 + ib : r0, d1 = LOWER ? r1 : s0;   // rows still to be updated
    if (d1 > d0)
      gemm(g, K, d1 - d0, nrhs, ib, -1.0, LU + (long long)s0 * nb + d0, nb, n2, 0, X + s0, nb, sX, true, X + d0, nb, sX);
  }
}

template <typename T> void lu_factor_t(Gemm& g, T* M, int nb, int K, int* perm, int* info, int* swp) {
  const long long n2 = (long long)nb * nb;
  constexpr int kOuter = Num<T>::NBLK;
  const int ss = lu_swap_ints(nb);
  const bool one = nb <= kOuter;   // one outer block: one list per matrix, applied to perm after every panel
  iota_rows<<<grid1((long long)nb * K), 256, 0, g.st>>>(perm, nb, K);
  for (int o0 = 0; o0 < nb; o0 += kOuter) {
    const int oend = nb - o0 < kOuter ? nb : o0 + kOuter, out = nb - (oend - o0) + 1, rest = nb - oend;
    int np = 0;
    for (int j0 = o0; j0 < oend; ++np) {
      int* lists = swp + np * kSwapInts;
      if (one) lists = swp;
      j0 += panel<T>(g, M, nb, K, o0, j0, oend, info, lists, ss);
      if (one) lu_swap_rest<T><<<dim3(1, K), 64, 0, g.st>>>(M, nb, o0, oend, 1, swp, ss, perm);
    }
    if (one) continue;
    lu_swap_rest<T><<<dim3((out + 63) / 64, K), 64, 0, g.st>>>(M, nb, o0, oend, np, swp, ss, perm);
    if (rest > 0) {
      // U12 = L11^{-1} A12, then A22 -= L21 U12
      solve_range<T, true>(g, M, nb, K, o0, oend, M + (long long)oend * nb, n2, rest, nullptr, 0);
      gemm(g, K, rest, rest, oend - o0, -1.0, M + (long long)o0 * nb + oend, nb, n2, 0, M + (long long)oend * nb + o0, nb, n2,
           true, M + (long long)oend * nb + oend, nb, n2);
    }
  }
  g.note(cudaGetLastError());
}

// A matrix of one block is solved by substitution alone, which needs no split
template <typename T> int solve_split(int nb, int split) { return nb <= Num<T>::NBLK ? 0 : split; }

template <typename T> void lu_solve_t(Gemm& g, const T* LU, int nb, int K, T* X, int nrhs, const T* dinv, int split) {
  const long long sx = (long long)nb * nrhs;
  split = solve_split<T>(nb, split);
  solve_range<T, true>(g, LU, nb, K, 0, nb, X, sx, nrhs, dinv, split);
  solve_range<T, false>(g, LU, nb, K, 0, nb, X, sx, nrhs, dinv, split);
  g.note(cudaGetLastError());
}

}  // namespace

int lu_swap_ints(int nb) { return nb <= 64 ? kSwapInts : kMaxPanels * kSwapInts; }

void lu_factor(Gemm& g, double2* M, int nb, int K, int* perm, int* info, int* swp) {
  lu_factor_t<double2>(g, M, nb, K, perm, info, swp);
}
void lu_factor(Gemm& g, float2* M, int nb, int K, int* perm, int* info, int* swp) {
  lu_factor_t<float2>(g, M, nb, K, perm, info, swp);
}
// Substitution costs 64 x 63 / 2 FP64 multiply-adds a column and block on the FP64 pipe (70-90 us a block for 400 to 512
// columns of 8 matrices), a product with the inverse about 25 us; the inverses of all blocks together cost one block's
// substitution.  For solves that are refined: one without refinement loses digits to the explicit inverses (lead_decimation_run).
// The line lies where gemm() slices the 64 x n x 64 products, at 2000 columns over the batch.  Measured above it, substitution /
// inverses: Dyson step of 8 x 512 rows (4096 columns) 11.8 / 9.9 ms, of 8 x 240 rows with two interior planes (3840) 5.6 / 4.6 ms.
const double2* lu_inverses(Gemm& g, const double2* LU, int nb, int K, int nrhs, int split) {
  constexpr int NB = Num<double2>::NBLK;
  if (!g.h || (double)nrhs * K * NB * NB < kSliceMin || nb < NB || (nb == NB && split > 0)) return nullptr;
  const int nblk = RowBlocks(nb, NB, split).count();
  if (nblk > 32767) return nullptr;
  void* w = nullptr;
  if (handle_ensure(g.h, 10, (size_t)K * nblk * 2 * NB * NB * sizeof(double2), &w) != RSFD_OK) return nullptr;
  lu_invert<<<dim3(NB / 4, K, 2 * nblk), 32, 0, g.st>>>(LU, nb, split, (double2*)w);
  g.note(cudaGetLastError());
  return (const double2*)w;
}
void lu_solve(Gemm& g, const double2* LU, int nb, int K, double2* X, int nrhs, const double2* dinv, int split) {
  lu_solve_t<double2>(g, LU, nb, K, X, nrhs, dinv, split);
}
void lu_solve(Gemm& g, const float2* LU, int nb, int K, float2* X, int nrhs, int split) {
  lu_solve_t<float2>(g, LU, nb, K, X, nrhs, nullptr, split);
}

void lu_permute(Gemm& g, const double2* B, int nb, int K, const int* perm, float2* X, int nrhs) {
  permute_rows<double2, float2><<<grid1((long long)nb * nrhs * K), 256, 0, g.st>>>(B, nb, nrhs, perm, X, K);
  g.note(cudaGetLastError());
}

void lu_permute(Gemm& g, const double2* B, int nb, int K, const int* perm, double2* X, int nrhs) {
  if (B != X) {
    permute_rows<double2, double2><<<grid1((long long)nb * nrhs * K), 256, 0, g.st>>>(B, nb, nrhs, perm, X, K);
    g.note(cudaGetLastError());
    return;
  }
  const size_t smem = (size_t)nb * sizeof(double2);
  if (smem <= 216 * 1024) {
    g.note(cudaFuncSetAttribute(permute_rows_inplace, cudaFuncAttributeMaxDynamicSharedMemorySize, 216 * 1024));
    permute_rows_inplace<<<dim3(nrhs, K), nb < 256 ? 64 : 256, smem, g.st>>>(X, nb, nrhs, perm);
    g.note(cudaGetLastError());
    return;
  }
  // taller columns: through a copy of a few columns at a time
  const int cols = 64;
  void* w = nullptr;
  if (!g.h || handle_ensure(g.h, 8, (size_t)nb * cols * sizeof(double2), &w) != RSFD_OK) {
    g.note(cudaErrorMemoryAllocation);
    return;
  }
  for (int b = 0; b < K; ++b)
    for (int c0 = 0; c0 < nrhs; c0 += cols) {
      const int nc = nrhs - c0 < cols ? nrhs - c0 : cols;
      double2* x = X + ((long long)b * nrhs + c0) * nb;
      g.note(cudaMemcpyAsync(w, x, (size_t)nb * nc * sizeof(double2), cudaMemcpyDeviceToDevice, g.st));
      permute_rows<double2, double2><<<grid1((long long)nb * nc), 256, 0, g.st>>>((const double2*)w, nb, nc,
                                                                                perm + (long long)b * nb, x, 1);
    }
  g.note(cudaGetLastError());
}

}  // namespace rsfd
