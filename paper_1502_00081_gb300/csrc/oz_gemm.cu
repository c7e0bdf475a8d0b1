// Complex FP64 GEMM on the tensor cores by error-free slicing (the scheme of Ozaki, Ogita, Oishi and
// Rump, "Error-free transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 59, 2012), for the Dyson step, the
// transmission and the lead decimation, whose matrix products are FP64.
//
// Why: the FP64 pipe of this GPU does about 0.5e12 FMA/s, 1/68 of its FP32 rate and 1/2000 of its
// 16-bit tensor rate, and those products were 85-97 % of the Dyson step.
//
// Arithmetic.  Every row of A (column of B) is scaled by a power of two so that its largest component
// is below 1 and written as a 62-bit fixed-point integer X = rint(x 2^62); X is cut into 8 balanced
// base-256 digits in [-128, 127] (the leading one within +-64), which are exact in bf16.  A product of
// digits is at most 2^14 (2^13 with a leading one), so the tensor core's FP32 sums are exact up to 2^24.
// Digit pairs (i, j), i, j = 0 .. 7, of equal weight 256^-(i+j) share an accumulator; pairs with i + j <= 7 are kept
// (36 of 64).  The accumulators are emptied every 128 complex k (256 real products): the sums of weights 0 .. 4
// are then at most 2^24 and exact; those of weights 5, 6 and 7 can reach 1.25, 1.5 and 1.75 x 2^24 (all digits near
// -128, all products of one sign), where every MMA that adds beyond 2^24 may lose up to 2 units of the weight.  The sums
// are added to 64-bit integers, so the k-sum has no further rounding, and the result is rounded to FP64 once.
// Error, in units of the row's scale times the column's (each at most twice the largest component): 7 x 2^-62 per real
// product from the dropped pairs, 2^-62 from the fixed point, and, only where a sum passes 2^24, up to 20 x 2 x 2^-52 per 128
// complex k from weight 5 (2^-54.7 per real product).  It is a bound relative to the largest element of the row and of
// the column, not to each element: elements below 2^-9 of their row's (column's) largest lose bits below 2^-63 of it.
// Callers whose sums mix parts of very different size cut the k-range between them (dense.cuh).
// FP32 operands take 30 bits and 4 digits, 10 pairs: all sums exact, 3 x 2^-30 per real product from the dropped pairs.
//
// Kernel.  One CTA per SM works through 128 x 32 tiles of complex C: eight accumulators of 128 x 32 for Re and eight for
// Im fill the 512 columns of tensor memory.  The digit planes are laid out in global memory exactly as
// the tensor core wants them in shared memory (K-major core matrices, no swizzle), so a k-step of 16
// is three contiguous bulk copies: one plane of A (8 digits x 128 rows, 32 KB), the other, and both
// planes of B (8 digits x 32 columns each, 16 KB).  The 8 digits of B are stacked along N, so digit i of A
// meets digits 1..9-i of B in ONE MMA of N = 32 (9 - i) whose columns fall onto the accumulators of
// weights i-1..7.  18 warps: 16 read the accumulators, one thread of the 17th issues the copies,
// one thread of the 18th the MMAs.
//
// Bound: tensor rate (144 real bf16 MACs per complex FP64 MAC, 40 per FP32 one; 36 B per clock and SM of operands from L2
// at full rate).  Measured: 16 products of 1024^3 in 4.0 ms, 4.3e12 complex multiply-adds/s, 1.24 PFLOP/s of bf16 MMAs = 0.64
// of the measured cuBLAS bf16 burst, tensor pipe active in 55 % of the cycles (132 ms on the FP64 pipe, 1.3e11/s).  One tile per CTA instead of a persistent CTA, so
// that a tile's set-up and write-back are not hidden: 4.6 ms, and 157 instead of 96 us for the FP32 LU's k = 128 updates.

#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "rsfd_internal.cuh"

namespace rsfd {
namespace {

// digits per element: 8 for FP64 operands, 4 for FP32 operands
template <typename T> struct OzOf;
template <> struct OzOf<double2> { static constexpr int S = 8, NA = 5; };
template <> struct OzOf<float2> { static constexpr int S = 4, NA = 10; };

constexpr int OZ_BM = 128;                    // rows of C per CTA
constexpr int OZ_KS = 16;                     // complex k per step (one MMA depth)
constexpr int OZ_CHUNK = 8;                   // k-steps between two emptyings of the accumulators
constexpr int OZ_NB = 3;                      // ring of B blocks
constexpr int OZ_BPLANE = 256 * OZ_KS * 2;    // bytes of one plane of B per k-step: digits x columns = 256 rows
constexpr int OZ_BBLK = 2 * OZ_BPLANE;
constexpr int OZ_EPI = 512;                   // epilogue threads (16 warps: 64 accumulator registers each)
constexpr int OZ_THREADS = OZ_EPI + 64;
template <int S> struct OzDim {
  static constexpr int BN = 256 / S;                 // columns of C per CTA
  static constexpr int EC = BN / (OZ_EPI / 128);     // columns per epilogue thread
  static constexpr int ABLK = S * OZ_BM * OZ_KS * 2; // bytes of one plane of A per k-step
};
template <typename T> constexpr int oz_smem() {
  return OzOf<T>::NA * OzDim<OzOf<T>::S>::ABLK + OZ_NB * OZ_BBLK + 1024;
}
constexpr uint32_t OZ_SBO = 128;
constexpr uint32_t OZ_LBO_A = (OZ_BM / 8) * 128;
constexpr uint32_t OZ_LBO_B = (256 / 8) * 128;
constexpr int kOzWaitCap = 1 << 12;           // attempts of a bounded wait, each up to 1 ms
constexpr uint32_t kOzHintNs = 1000000;

__device__ __forceinline__ uint32_t oz_saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// one attempt, up to 1 ms
__device__ __forceinline__ bool oz_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(kOzHintNs)
      : "memory");
  return ok != 0;
}
// bounded wait; also gives up when another thread has (looked at between attempts only: a role that goes on for a while
// does no harm, it soon waits for the one that stopped)
__device__ __forceinline__ bool oz_wait(uint32_t bar, uint32_t parity, int cap, const volatile int& abort) {
  for (int i = 0; i < cap; ++i) {
    if (oz_try(bar, parity)) return true;
    if (abort) return false;
  }
  return false;
}
// bounded wait for what is in flight (after an abort, before the CTA's memory is given back)
__device__ __forceinline__ void oz_drain(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < kOzWaitCap && !oz_try(bar, parity); ++i) {
  }
}
__device__ __forceinline__ void oz_bulk(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ uint64_t oz_desc(uint32_t saddr, uint32_t lbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((OZ_SBO >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}
// kind::f16 instruction descriptor: FP32 accumulator, bf16 A and B, both K-major, M = 128
__host__ __device__ constexpr uint32_t oz_idesc(int N, int negA) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)negA << 13) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(OZ_BM >> 4) << 24);
}
__device__ __forceinline__ void oz_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void oz_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void oz_tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// one operand: element (row, k) of matrix b at p[b sb + row rs + k ks] (row: a row of op(A) or a column of B)
template <typename T> struct OzOperand {
  const T* p;
  long long sb, rs, ks;
  int rows;         // m or n
  int conj;
  int is_b;
  unsigned int* ex;     // [batch][rows_pad] high words of the largest component
  unsigned char* dig;   // digit planes
  int rows_pad;
};
template <typename T> struct OzSplit {
  OzOperand<T> o[2];
  int k, ksteps, batch;
};

// sign-cleared leading word of a component: ordered like its magnitude
__device__ __forceinline__ unsigned oz_word(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ unsigned oz_word(float x) { return __float_as_uint(x) & 0x7fffffffu; }
template <typename T> __device__ __forceinline__ unsigned oz_word2(T v) { return max(oz_word(v.x), oz_word(v.y)); }
// words of infinities and NaN start here
template <typename T> __host__ __device__ constexpr unsigned oz_nonfinite() { return sizeof(T) == 16 ? 0x7ff00000u : 0x7f800000u; }

// Largest component of every row: leading words compared as integers.  Rows contiguous in memory
// (rs = 1): a thread per row; k contiguous: a warp per row.  Bound: one read of the operand.
template <typename T> __global__ void __launch_bounds__(256) oz_rowmax(OzSplit<T> q) {
  const OzOperand<T>& o = q.o[blockIdx.z & 1];
  const int b = blockIdx.z >> 1;
  const T* p = o.p + b * o.sb;
  if (o.ks != 1) {
    const int row = blockIdx.x * 32 + (threadIdx.x & 31);
    unsigned int m = 0;
    if (row < o.rows)
      for (int k = blockIdx.y * 64 + (threadIdx.x >> 5); k < min(q.k, (int)blockIdx.y * 64 + 64); k += 8)
        m = max(m, oz_word2(p[row * o.rs + k * o.ks]));
    __shared__ unsigned int s[8][32];
    s[threadIdx.x >> 5][threadIdx.x & 31] = m;
    __syncthreads();
    if (threadIdx.x < 32 && row < o.rows) {
#pragma unroll
      for (int w = 1; w < 8; ++w) m = max(m, s[w][threadIdx.x]);
      atomicMax(o.ex + (size_t)b * o.rows_pad + row, m);
    }
  } else {
    // 32 rows per block, a warp takes 4 of them
    for (int r = threadIdx.x >> 5; r < 32; r += 8) {
      const int row = blockIdx.x * 32 + r;
      if (row >= o.rows) break;
      unsigned int m = 0;
      for (int k = blockIdx.y * 64 + (threadIdx.x & 31); k < min(q.k, (int)blockIdx.y * 64 + 64); k += 32)
        m = max(m, oz_word2(p[row * o.rs + k]));
      m = __reduce_max_sync(0xffffffffu, m);
      if ((threadIdx.x & 31) == 0) atomicMax(o.ex + (size_t)b * o.rows_pad + row, m);
    }
  }
}

// binary exponent se with |x| < 2^se for every component of a row whose largest leading word is w
template <typename T> __device__ __forceinline__ int oz_exponent(unsigned int w) {
  const int e = (int)(w >> (sizeof(T) == 16 ? 20 : 23));
  return (e < 1 ? 1 : e) - (sizeof(T) == 16 ? 1022 : 126);
}

// fixed point rint(x 2^(62 - se)) (FP64) or rint(x 2^(30 - se)) (FP32), integer arithmetic only
__device__ __forceinline__ long long oz_fixed(double x, int se) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((u >> 52) & 0x7ff);
  unsigned long long m = u & 0xfffffffffffffull;
  if (e > 0) m |= 1ull << 52;
  const int sh = (e < 1 ? 1 : e) - 1075 - se + 62;   // at most 9
  if (sh >= 0) m <<= sh;
  else m = sh > -62 ? (m + (1ull << (-sh - 1))) >> (-sh) : 0ull;
  return (u >> 63) ? -(long long)m : (long long)m;
}
__device__ __forceinline__ int oz_fixed(float x, int se) {
  const unsigned u = __float_as_uint(x);
  const int e = (int)((u >> 23) & 0xff);
  unsigned m = u & 0x7fffffu;
  if (e > 0) m |= 1u << 23;
  const int sh = (e < 1 ? 1 : e) - 150 - se + 30;    // at most 6
  if (sh >= 0) m <<= sh;
  else m = sh > -30 ? (m + (1u << (-sh - 1))) >> (-sh) : 0u;
  return (u >> 31) ? -(int)m : (int)m;
}

// Digit planes.  A thread takes 8 consecutive k of one row: 8 loads, then one 16-byte store per digit and
// plane (consecutive rows are 16 bytes apart, so a warp stores 512 contiguous bytes).
// Bound: the stores (4 bytes per digit and element) and one read.
template <typename T> __global__ void __launch_bounds__(256) oz_digits(OzSplit<T> q) {
  constexpr int S = OzOf<T>::S, BN = OzDim<S>::BN, ABLK = OzDim<S>::ABLK;
  typedef decltype(oz_fixed(T().x, 0)) I;
  const OzOperand<T>& o = q.o[blockIdx.z & 1];
  const int b = blockIdx.z >> 1;
  const int row = blockIdx.x * 32 + (threadIdx.x & 31);
  const int kg = blockIdx.y * 8 + (threadIdx.x >> 5);   // group of 8 k
  if (row >= o.rows_pad || kg >= 2 * q.ksteps) return;
  const T* p = o.p + b * o.sb + (long long)row * o.rs;
  const int se = row < o.rows ? oz_exponent<T>(o.ex[(size_t)b * o.rows_pad + row]) : 0;
  I xr[8], xi[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const int k = kg * 8 + t;
    T v = T();
    if (row < o.rows && k < q.k) v = p[k * o.ks];
    if (o.conj) v.y = -v.y;
    xr[t] = oz_fixed(v.x, se);
    xi[t] = oz_fixed(v.y, se);
  }
  const int ks = kg >> 1, kh = kg & 1;
  unsigned char *d0, *d1;   // digit 0 (leading) of the two planes
  uint32_t step;            // bytes from one digit to the next
  if (o.is_b) {
    const int nt = row / BN, r = row % BN;
    unsigned char* blk = o.dig + (((size_t)b * (o.rows_pad / BN) + nt) * q.ksteps + ks) * OZ_BBLK;
    d0 = blk + kh * OZ_LBO_B + r * 16;      // stacked row = digit * BN + r
    d1 = d0 + OZ_BPLANE;
    step = BN * 16;
  } else {
    const int mt = row / OZ_BM, r = row % OZ_BM;
    unsigned char* blk = o.dig + (((size_t)b * (o.rows_pad / OZ_BM) + mt) * q.ksteps + ks) * (2 * ABLK);
    d0 = blk + kh * OZ_LBO_A + r * 16;
    d1 = d0 + ABLK;
    step = OZ_BM * OZ_KS * 2;
  }
#pragma unroll
  for (int s = S - 1; s >= 0; --s) {
    uint32_t wr[4], wi[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      float f[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        I &a = xr[2 * t + h], &c = xi[2 * t + h];
        const int da = s > 0 ? (int)(signed char)(a & 0xff) : (int)a;
        const int dc = s > 0 ? (int)(signed char)(c & 0xff) : (int)c;
        a = (a - da) >> 8;
        c = (c - dc) >> 8;
        f[h] = (float)da;
        f[2 + h] = (float)dc;
      }
      asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(wr[t]) : "f"(f[1]), "f"(f[0]));
      asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(wi[t]) : "f"(f[3]), "f"(f[2]));
    }
    *(uint4*)(d0 + (size_t)s * step) = make_uint4(wr[0], wr[1], wr[2], wr[3]);
    *(uint4*)(d1 + (size_t)s * step) = make_uint4(wi[0], wi[1], wi[2], wi[3]);
  }
}

template <typename T> struct OzGemm {
  const unsigned char *A, *B;
  const unsigned int *exA, *exB;
  int m, n, m_pad, n_pad, ksteps;
  int tiles;          // 128 x BN tiles of all matrices
  int sign;           // alpha (+1 or -1)
  int add;            // 1: add C
  T* C;
  int ldc;
  long long sC;
  int* err;
  int cap;            // attempts of a bounded wait
};

// (hi 2^32 + lo) 2^e rounded to nearest, by integer arithmetic (conversions and FP64 arithmetic run at 2 a
// clock and SM): FP64 result of the 8-digit form
__device__ __forceinline__ double oz_round(long long hi, long long lo, int e) {
  long long h = hi + (lo >> 32);
  unsigned l = (unsigned)lo;
  const bool neg = h < 0;
  if (neg) {
    h = -h - (l != 0u);
    l = 0u - l;
  }
  unsigned long long m;     // leading 64 bits of the magnitude, top bit at 63
  int x;                    // value = m 2^x (bits below m only matter as a rounding tie and are dropped)
  if (h != 0) {
    const int z = __clzll(h);
    m = (unsigned long long)h << z;
    if (z <= 32) m |= (unsigned long long)l >> (32 - z);
    else m |= (unsigned long long)l << (z - 32);
    x = 32 - z;
  } else {
    if (l == 0u) return 0.0;
    const int z = __clz(l);
    m = (unsigned long long)l << (32 + z);
    x = -32 - z;
  }
  const int ex = x + e + 63 + 1023;   // biased exponent of the leading bit
  if (ex <= 0 || ex >= 2046) {        // near the ends of the range: the library's scaling
    const double v = scalbn((double)m, x + e);
    return neg ? -v : v;
  }
  // 53 bits, round half up; a carry out of the mantissa raises the exponent field by itself
  const unsigned long long r = (m + 0x400ull) >> 11;
  const unsigned long long bits = r < (1ull << 52) ? ((unsigned long long)(ex + 1) << 52)   // m + 0x400 wrapped
                                                   : ((unsigned long long)(ex - 1) << 52) + r;
  return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0ull)));
}
// FP32 result of the 4-digit form: hi 2^e
__device__ __forceinline__ float oz_round(long long hi, int e) {
  const int h = (int)(hi >> 32);
  const unsigned l = (unsigned)hi;
  return scalbnf(fmaf((float)h, 0x1p32f, (float)l), e);
}

template <typename T> __global__ void __launch_bounds__(OZ_THREADS, 1) oz_gemm_kernel(OzGemm<T> q) {
  constexpr int S = OzOf<T>::S, NA = OzOf<T>::NA, BN = OzDim<S>::BN, EC = OzDim<S>::EC, ABLK = OzDim<S>::ABLK;
  constexpr int SW = S / 4;   // 64-bit sums per component
  extern __shared__ __align__(1024) unsigned char oz_smem_raw[];
  __shared__ __align__(8) uint64_t fullA[NA], emptyA[NA], fullB[OZ_NB], emptyB[OZ_NB], accFull, accEmpty, mmaDone;
  __shared__ uint32_t tmem_s;
  __shared__ volatile int s_abort;
  __shared__ int s_issuedA, s_issuedB;   // copies issued (read after an abort)
  unsigned char* smem = (unsigned char*)(((uintptr_t)oz_smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* sA = smem;
  unsigned char* sB = smem + NA * ABLK;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int mtiles = q.m_pad / OZ_BM, ntiles = q.n_pad / BN;
  // tile t: row tile fastest, then column tile, then matrix
  auto decode = [&](int t, int& mt, int& nt, int& b) {
    mt = t % mtiles;
    const int r = t / mtiles;
    nt = r % ntiles;
    b = r / ntiles;
  };
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(oz_saddr(&tmem_s)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    auto init = [](uint64_t* bar, int count) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(oz_saddr(bar)), "r"(count) : "memory");
    };
    for (int i = 0; i < NA; ++i) {
      init(&fullA[i], 1);
      init(&emptyA[i], 1);
    }
    for (int i = 0; i < OZ_NB; ++i) {
      init(&fullB[i], 1);
      init(&emptyB[i], 1);
    }
    init(&accFull, 1);
    init(&mmaDone, 1);
    init(&accEmpty, OZ_EPI);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_s;
  const int ksteps = q.ksteps;
  const int nchunks = (ksteps + OZ_CHUNK - 1) / OZ_CHUNK;

  if (warp == OZ_EPI / 32) {
    // copies: per k-step B (both planes), then the two planes of A; ring positions run on over the tiles
    if (lane == 0) {
      bool ok = true;
      int issuedA = 0, issuedB = 0;
      for (int tile = blockIdx.x; tile < q.tiles && ok; tile += gridDim.x) {
        int mt, nt, b;
        decode(tile, mt, nt, b);
        const unsigned char* gA = q.A + ((size_t)b * mtiles + mt) * ksteps * (2 * ABLK);
        const unsigned char* gB = q.B + ((size_t)b * ntiles + nt) * ksteps * OZ_BBLK;
        for (int t = 0; t < ksteps && ok; ++t) {
          const int sb = issuedB % OZ_NB;
          ok = issuedB < OZ_NB || oz_wait(oz_saddr(&emptyB[sb]), (uint32_t)((issuedB / OZ_NB - 1) & 1), q.cap, s_abort);
          if (!ok) break;
          oz_bulk(oz_saddr(sB + sb * OZ_BBLK), gB + (size_t)t * OZ_BBLK, OZ_BBLK, oz_saddr(&fullB[sb]));
          ++issuedB;
          for (int h = 0; h < 2; ++h) {
            const int sa = issuedA % NA;
            ok = issuedA < NA || oz_wait(oz_saddr(&emptyA[sa]), (uint32_t)((issuedA / NA - 1) & 1), q.cap, s_abort);
            if (!ok) break;
            oz_bulk(oz_saddr(sA + sa * ABLK), gA + (size_t)(2 * t + h) * ABLK, ABLK, oz_saddr(&fullA[sa]));
            ++issuedA;
          }
        }
      }
      s_issuedA = issuedA;
      s_issuedB = issuedB;
      if (!ok) {
        s_abort = 1;
        atomicExch(q.err, 1);
      }
    }
  } else if (warp == OZ_EPI / 32 + 1) {
    if (lane == 0) {
      bool ok = true;
      int ia = 0, ib = 0, cc = 0;   // planes of A, blocks of B and chunks so far
      for (int tile = blockIdx.x; tile < q.tiles && ok; tile += gridDim.x) {
        for (int t = 0; t < ksteps && ok; ++t) {
          const bool first = t % OZ_CHUNK == 0;
          if (first && cc > 0) {   // the accumulators have been read
            ok = oz_wait(oz_saddr(&accEmpty), (uint32_t)((cc - 1) & 1), q.cap, s_abort);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          const int sb = ib % OZ_NB;
          ok = ok && oz_wait(oz_saddr(&fullB[sb]), (uint32_t)((ib / OZ_NB) & 1), q.cap, s_abort);
          const uint32_t b0 = oz_saddr(sB + sb * OZ_BBLK);
          const uint64_t bre = oz_desc(b0, OZ_LBO_B), bim = oz_desc(b0 + OZ_BPLANE, OZ_LBO_B);
          for (int h = 0; h < 2 && ok; ++h) {
            const int sa = ia % NA;
            ok = oz_wait(oz_saddr(&fullA[sa]), (uint32_t)((ia / NA) & 1), q.cap, s_abort);
            if (!ok) break;
            const uint32_t a0 = oz_saddr(sA + sa * ABLK);
            // h = 0: Re += Ar Br, Im += Ar Bi;  h = 1: Re -= Ai Bi, Im += Ai Br
#pragma unroll
            for (int i = 0; i < S; ++i) {
              const uint64_t ad = oz_desc(a0 + i * (OZ_BM * OZ_KS * 2), OZ_LBO_A);
              const uint32_t acc = (first && h == 0 && i == 0) ? 0u : 1u;
              const int N = BN * (S - i);
              oz_mma(tmem + i * BN, ad, h ? bim : bre, h ? oz_idesc(N, 1) : oz_idesc(N, 0), acc);
              oz_mma(tmem + 256 + i * BN, ad, h ? bre : bim, oz_idesc(N, 0), acc);
            }
            oz_commit(oz_saddr(&emptyA[sa]));
            ++ia;
          }
          if (!ok) break;
          oz_commit(oz_saddr(&emptyB[sb]));
          ++ib;
          if (t % OZ_CHUNK == OZ_CHUNK - 1 || t == ksteps - 1) {
            oz_commit(oz_saddr(&accFull));
            ++cc;
          }
        }
      }
      if (!ok) {
        // the MMAs issued so far end before the tensor memory is given back
        s_abort = 1;
        atomicExch(q.err, 1);
        if (ia > 0) {
          oz_commit(oz_saddr(&mmaDone));
          oz_drain(oz_saddr(&mmaDone), 0);
        }
      }
    }
  } else {
    // epilogue threads: row 32 (warp % 4) + lane, columns EC (warp / 4) ... of Re and of Im
    const int ch = (warp >> 2) * EC;
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16) + ch;
    bool ok = true;
    int cc = 0;   // chunks so far
    // the sums of a tile are written while the next tile's MMAs run: they only wait for the accumulators to be read
    for (int tile = blockIdx.x; tile < q.tiles && ok; tile += gridDim.x) {
    long long sum[2][SW][EC];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int w = 0; w < SW; ++w)
#pragma unroll
        for (int j = 0; j < EC; ++j) sum[p][w][j] = 0;
    for (int c = 0; c < nchunks; ++c, ++cc) {
      // the warp goes on or stops as a whole: what follows is warp-aligned
      ok = __all_sync(0xffffffffu, oz_wait(oz_saddr(&accFull), (uint32_t)(cc & 1), q.cap, s_abort));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int p = 0; p < 2; ++p) {
#pragma unroll
        for (int d = 0; d < S; d += 2) {
#pragma unroll
          for (int j0 = 0; j0 < EC; j0 += 8) {
            uint32_t r0[8], r1[8];
            oz_tmem_ld8(tl + p * 256 + d * BN + j0, r0);
            oz_tmem_ld8(tl + p * 256 + (d + 1) * BN + j0, r1);
            // the registers pass through the wait so that no use moves above it
            asm volatile("tcgen05.wait::ld.sync.aligned;"
                         : "+r"(r0[0]), "+r"(r0[1]), "+r"(r0[2]), "+r"(r0[3]), "+r"(r0[4]), "+r"(r0[5]), "+r"(r0[6]),
                           "+r"(r0[7]), "+r"(r1[0]), "+r"(r1[1]), "+r"(r1[2]), "+r"(r1[3]), "+r"(r1[4]), "+r"(r1[5]),
                           "+r"(r1[6]), "+r"(r1[7])
                         :
                         : "memory");
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              long long& acc = sum[p][d / 4][j0 + j];
              acc += (long long)__float2int_rn(__uint_as_float(r0[j])) * (1ll << (8 * (3 - (d & 3))));
              acc += (long long)__float2int_rn(__uint_as_float(r1[j])) * (1ll << (8 * (2 - (d & 3))));
            }
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(oz_saddr(&accEmpty)) : "memory");
    }
    int mt, nt, b;
    decode(tile, mt, nt, b);
    const int row = mt * OZ_BM + (warp & 3) * 32 + lane;
    if (ok && row < q.m) {
      const unsigned int wa = q.exA[(size_t)b * q.m_pad + row];
      const int ea = oz_exponent<T>(wa);
#pragma unroll
      for (int j = 0; j < EC; ++j) {
        const int col = nt * BN + ch + j;
        if (col < q.n) {
          const unsigned int wb = q.exB[(size_t)b * q.n_pad + col];
          const int e = ea + oz_exponent<T>(wb);
          T v;
          if constexpr (S == 8) {
            v.x = oz_round(sum[0][0][j], sum[0][SW - 1][j], e - 68);
            v.y = oz_round(sum[1][0][j], sum[1][SW - 1][j], e - 68);
          } else {
            v.x = oz_round(sum[0][0][j], e - 36);
            v.y = oz_round(sum[1][0][j], e - 36);
          }
          if (wa >= oz_nonfinite<T>() || wb >= oz_nonfinite<T>()) v.x = v.y = CUDART_NAN_F;
          T* cp = q.C + b * q.sC + (long long)col * q.ldc + row;
          T o = T();
          if (q.add) o = *cp;
          if (q.sign < 0) {
            o.x -= v.x;
            o.y -= v.y;
          } else {
            o.x += v.x;
            o.y += v.y;
          }
          *cp = o;
        }
      }
    }
    }
    if (!ok) {
      s_abort = 1;
      atomicExch(q.err, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  if (s_abort) {
    // the copies in flight land before the CTA's shared memory is released: per ring entry the last one issued (earlier
    // ones completed before the entry was refilled)
    if (tid == 0) {
      for (int a = max(0, s_issuedA - NA); a < s_issuedA; ++a) oz_drain(oz_saddr(&fullA[a % NA]), (uint32_t)((a / NA) & 1));
      for (int c = max(0, s_issuedB - OZ_NB); c < s_issuedB; ++c)
        oz_drain(oz_saddr(&fullB[c % OZ_NB]), (uint32_t)((c / OZ_NB) & 1));
    }
    __syncthreads();
  }
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

size_t up(size_t x, size_t a) { return (x + a - 1) / a * a; }

template <typename T> size_t oz_bytes_t(int m, int n, int k) {
  constexpr int S = OzOf<T>::S;
  const size_t mp = up(m, OZ_BM), np = up(n, OzDim<S>::BN), ks = (k + OZ_KS - 1) / OZ_KS;
  return mp / OZ_BM * ks * 2 * OzDim<S>::ABLK + np / OzDim<S>::BN * ks * OZ_BBLK + up((mp + np) * sizeof(unsigned int), 256);
}

template <typename T>
cudaError_t oz_gemm_t(cudaStream_t st, int batch, int m, int n, int k, int sign, const T* A, int lda, long long sA,
                      int opA, const T* B, int ldb, long long sB, int add, T* C, int ldc, long long sC, void* work,
                      size_t work_bytes, int* err, int wait_cap) {
  constexpr int S = OzOf<T>::S, BN = OzDim<S>::BN, ABLK = OzDim<S>::ABLK;
  const size_t per = oz_bytes_t<T>(m, n, k);
  int nb = (int)(work_bytes / per < (size_t)batch ? work_bytes / per : (size_t)batch);
  if (nb < 1) return cudaErrorInvalidValue;
  if (nb > 32767) nb = 32767;   // gridDim.z carries (matrix, operand)
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int mp = (int)up(m, OZ_BM), np = (int)up(n, BN), ks = (k + OZ_KS - 1) / OZ_KS;
  cudaError_t e = cudaFuncSetAttribute(oz_gemm_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, oz_smem<T>());
  if (e != cudaSuccess) return e;
  for (int b0 = 0; b0 < batch; b0 += nb) {
    const int bn = batch - b0 < nb ? batch - b0 : nb;
    unsigned char* dA = (unsigned char*)work;
    unsigned char* dB = dA + (size_t)bn * (mp / OZ_BM) * ks * 2 * ABLK;
    unsigned int* xA = (unsigned int*)(dB + (size_t)bn * (np / BN) * ks * OZ_BBLK);
    unsigned int* xB = xA + (size_t)bn * mp;
    OzSplit<T> q;
    q.k = k;
    q.ksteps = ks;
    q.batch = bn;
    q.o[0] = OzOperand<T>{A + b0 * sA, sA, opA ? lda : 1, opA ? 1 : lda, m, opA, 0, xA, dA, mp};
    q.o[1] = OzOperand<T>{B + b0 * sB, sB, ldb, 1, n, 0, 1, xB, dB, np};
    e = cudaMemsetAsync(xA, 0, (size_t)bn * (mp + np) * sizeof(unsigned int), st);
    if (e != cudaSuccess) return e;
    const int rows = m > n ? m : n, rpad = mp > np ? mp : np;
    oz_rowmax<T><<<dim3((rows + 31) / 32, (k + 63) / 64, 2 * bn), 256, 0, st>>>(q);
    oz_digits<T><<<dim3((rpad + 31) / 32, (2 * ks + 7) / 8, 2 * bn), 256, 0, st>>>(q);
    const long long tiles = (long long)(mp / OZ_BM) * (np / BN) * bn;
    if (tiles > 0x7fffffffll) return cudaErrorInvalidValue;
    OzGemm<T> g{dA, dB, xA, xB, m, n, mp, np, ks, (int)tiles, sign, add, C + b0 * sC, ldc, sC, err,
                wait_cap == 0 ? kOzWaitCap : (wait_cap < 0 ? 0 : wait_cap)};
    oz_gemm_kernel<T><<<(int)(tiles < sms ? tiles : sms), OZ_THREADS, oz_smem<T>(), st>>>(g);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

size_t oz_bytes(int m, int n, int k, bool fp64) {
  return fp64 ? oz_bytes_t<double2>(m, n, k) : oz_bytes_t<float2>(m, n, k);
}

cudaError_t oz_gemm(cudaStream_t st, int batch, int m, int n, int k, int sign, const double2* A, int lda, long long sA,
                    int opA, const double2* B, int ldb, long long sB, int add, double2* C, int ldc, long long sC,
                    void* work, size_t work_bytes, int* err, int wait_cap) {
  return oz_gemm_t<double2>(st, batch, m, n, k, sign, A, lda, sA, opA, B, ldb, sB, add, C, ldc, sC, work, work_bytes, err,
                            wait_cap);
}
cudaError_t oz_gemm(cudaStream_t st, int batch, int m, int n, int k, int sign, const float2* A, int lda, long long sA,
                    int opA, const float2* B, int ldb, long long sB, int add, float2* C, int ldc, long long sC, void* work,
                    size_t work_bytes, int* err, int wait_cap) {
  return oz_gemm_t<float2>(st, batch, m, n, k, sign, A, lda, sA, opA, B, ldb, sB, add, C, ldc, sC, work, work_bytes, err,
                           wait_cap);
}

}  // namespace rsfd
