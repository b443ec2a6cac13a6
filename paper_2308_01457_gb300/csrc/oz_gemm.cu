// FP64-class complex GEMM C <- beta C + alpha Z X on the bf16 tensor cores by exact digit
// splitting, for the refinement residuals of multi-right-hand-side solves (A6, A9).
//
// Every row i of Z is scaled by a power of two sigma_i > its largest |Re|, |Im| and written
// as seven signed base-256 digits:  Z_ik = sigma_i 2^-7 sum_{s=0..6} 2^{-8s} d_s[i,k] up to
// 2^-56 sigma_i (the balanced base-256 form of Z_ik 2^55 / sigma_i rounded to an integer),
// |d_s| <= 128, so each digit is exact in bf16; the same
// for every column j of X with tau_j and digits e_t.  Then
//   (Z X)_ij = sigma_i tau_j 2^-14 sum_{s,t} 2^{-8(s+t)} sum_k d_s[i,k] e_t[k,j],
// and a digit product is an integer of at most 2^14, so sums of the same order g = s+t over
// 128 values of k are exact in the FP32 accumulators of the tensor cores for g <= 3
// ((g+1) x 2 x 128 x 2^14 <= 2^24; order 4 too unless nearly all digits are at the ends of their range,
// the first ones included, and then its rounding is below 2^-49 of |Z||X|).  Orders g <= 6 (28 digit pairs) are kept: the dropped
// terms are below 2^-56 of sigma_i tau_j per product (the trailing updates of FP64 factorisations keep
// order 7 too, 34 pairs, and leave nothing of that size but the rounding of the operands).  After every
// 128 values of k the seven order accumulators are read out of TMEM: orders 0-4 are added into a 64-bit integer
// sum per output, orders 5-6 (below 2^-40 of them) into an FP32 sum; the result is scaled by
// sigma_i tau_j 2^-14.
//
// What bounds it is the issue of the MMAs and then the tensor pipe.  An MMA with M = 128, K = 16
// takes 44 cycles for any N up to 64 behind `lane == 0`, where its operands go from vector to
// uniform registers one by one; behind elect.sync, with every operand a compile-time offset, N = 64
// takes 35 (32 of them the pipe) and N = 32 takes 21 (measured).  So Re and Im are separate tiles
// of N = 64, seven orders of which fill 448 of the 512 TMEM columns, and the orders, the part and
// the stage are compiled in.  Every wait of the issuing lane costs 80 cycles even with nothing to
// wait for: one per step, tested ahead.  Z X at N = 7503 with 163 columns (354 half tiles over 152
// SMs): 4.63 ms with both parts at N = 32, sums after every 64 values of k and `lane == 0`; 2.24 ms
// with N = 64 and elect; 1.63 ms with one wait per step and a load lane per digit.  The MMAs alone
// take 1.22 ms (1968 cycles per step of 56), the order sums 0.25 ms, the rest is waiting for L2.
//
// Kernel roles (one CTA per SM, persistent over 128 x 64 tiles of one part): seven lanes of warp 0
// move the pre-tiled digits of a 16-wide k step into one of two stages with bulk copies, lane s
// digit s of Z (8 KB) as soon as its slot is free, lane 0 also all of X's (28 KB); one lane of warp
// 1 issues the 56 MMAs of a step (tcgen05.mma kind::f16, bf16, M = 128, N = 64, K = 16; the minus of
// Im Z Im X via the negate-B bit; the MMAs of an A tile run back to back and keep it in the A
// collector) into the order accumulators; warps 2-9 read the accumulators after every 128 values of
// k and hold the sums (two warps per TMEM lane group, 32 columns each).  All waits are bounded.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <thread>
#include <type_traits>

#include "fosb_internal.h"

namespace fosb {
namespace {

constexpr int OZ_TM = 128, OZ_TN = 64, OZ_KS = 16, OZ_ND = 7;  // tile rows, tile columns, k step, digits
constexpr int OZ_KCH = 8;                                      // k steps per chunk (128 values)
constexpr int OZ_ATILE = OZ_TM * OZ_KS * 2;                    // 4096 B
constexpr int OZ_BTILE = OZ_TN * OZ_KS * 2;                    // 2048 B
constexpr int OZ_NT = OZ_ND * 2;                               // digit x part tiles per operand and step
constexpr int OZ_ASLOT = 2 * OZ_ATILE;                         // one digit of Z (Re, Im)
constexpr int OZ_BSLOT = OZ_NT * OZ_BTILE;                     // all digits of X
constexpr int OZ_STAGE = OZ_ND * OZ_ASLOT + OZ_BSLOT;          // 86016 B, one k step
constexpr int OZ_SMEM = 2 * OZ_STAGE + 1024;
constexpr int OZ_THREADS = 10 * 32;                            // producer, MMA, 8 flush warps
constexpr int OZ_FLUSH = 8 * 32;
constexpr int OZ_HN = OZ_TN / 2;                               // columns per flush thread
constexpr int OZ_TMEM_COLS = 512;                              // 7 or 8 orders x 64 columns
constexpr long long kOzSpinLimit = 1ll << 24;
// Poll limit of the waits between the roles on this device (kOzSpinLimit unless changed by
// fosb_debug_set_wait_limit).  The waits for copies and MMAs in flight before the kernel leaves keep
// kOzSpinLimit.
__device__ long long g_oz_wait_limit = kOzSpinLimit;
static_assert(OZ_SMEM <= 226 * 1024, "digit stages and the barriers do not fit shared memory");

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// canonical no-swizzle K-major offset of element (row, k), k < 16, 2-byte elements:
// 8 x 16-byte core matrices, 128 B apart along k, 256 B between 8-row groups
__host__ __device__ __forceinline__ int oz_off(int row, int k) {
  return (row >> 3) * 256 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}
__device__ __forceinline__ uint64_t oz_desc(uint32_t addr) {
  const uint64_t lbo = 128, sbo = 256;
  return uint64_t((addr >> 4) & 0x3FFF) | (uint64_t((lbo >> 4) & 0x3FFF) << 16) |
         (uint64_t((sbo >> 4) & 0x3FFF) << 32) | (uint64_t(1) << 46);
}
// kind::f16 instruction descriptor: D f32 (bits 4-5 = 1), A and B bf16 (bits 7-9, 10-12 = 1),
// K-major A and B, N >> 3 at bits 17-22, M >> 4 at bits 24-28, optional negate-B (bit 14)
__host__ __device__ constexpr uint32_t oz_idesc(bool neg_b) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (neg_b ? (1u << 14) : 0u) | (uint32_t(OZ_TN >> 3) << 17) |
         (uint32_t(OZ_TM >> 4) << 24);
}
// One MMA; CU says what the A collector does: 0 = fill (read A, keep it), 1 = use the kept A,
// 2 = use it for the last time.  Consecutive MMAs on the same A tile read it from shared
// memory once.
__device__ __forceinline__ void oz_mma_once(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
}
template <int CU>
__device__ __forceinline__ void oz_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  if constexpr (CU == 0)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
  else if constexpr (CU == 1)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
  else
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
}
// One lane of a converged warp.  The compiler knows that the branch on it has one thread and keeps
// the MMA operands in uniform registers; behind `lane == 0` every MMA takes 44 cycles to issue.
__device__ __forceinline__ bool oz_elect() {
  uint32_t p;
  asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ uint32_t oz_test(uint32_t mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(mbar), "r"(parity)
      : "memory");
  return done;
}
template <bool SLEEP = false>
__device__ __forceinline__ bool oz_wait(uint32_t mbar, uint32_t parity, long long limit = kOzSpinLimit) {
  for (long long spins = 0; spins < limit; ++spins) {
    if (oz_test(mbar, parity)) return true;
    if (SLEEP) __nanosleep(32);
  }
  return false;
}
// barrier of the eight flush warps; true where any of their threads passed true
__device__ __forceinline__ bool oz_any(bool x) {
  uint32_t any;
  asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 q, %1, 0;\n bar.red.or.pred p, 1, 256, q;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(any)
               : "r"(uint32_t(x))
               : "memory");
  return any != 0;
}
__device__ __forceinline__ void oz_init(uint32_t a, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count));
}
__device__ __forceinline__ void oz_arrive(uint32_t a) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(a));
}
__device__ __forceinline__ void oz_expect_tx(uint32_t a, uint32_t bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(a), "r"(bytes));
}
__device__ __forceinline__ void oz_bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(mbar)
               : "memory");
}
__device__ __forceinline__ void oz_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar));
}
__device__ __forceinline__ void oz_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}
// waits for the loads above; the registers pass through, so that no use of them moves before it
__device__ __forceinline__ void oz_wait_ld(uint32_t (&v)[8], uint32_t (&u)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                 "+r"(u[0]), "+r"(u[1]), "+r"(u[2]), "+r"(u[3]), "+r"(u[4]), "+r"(u[5]), "+r"(u[6]), "+r"(u[7])
               :
               : "memory");
}

// ---------------------------------------------------------------- digit splitting
// |x| as an ordered integer: the bit pattern with the sign cleared (non-negative doubles
// compare like their bit patterns), so the maxima below run on the integer pipe.
__device__ __forceinline__ unsigned long long oz_abs_bits(double x) {
  return static_cast<unsigned long long>(__double_as_longlong(x)) & 0x7FFFFFFFFFFFFFFFull;
}
// the smallest e with |x| < 2^e for the largest |x| of a row or column (bit pattern mb),
// e = 0 for zero: m = f 2^e with f in [0.5, 1)
// Rows and columns with an infinity or NaN have the exponent OZ_BAD and give NaN.
constexpr int OZ_BAD = 1 << 28;
__device__ __forceinline__ int oz_exponent(unsigned long long mb) {
  int e = 0;
  if (mb >= 0x7FF0000000000000ull) e = OZ_BAD;
  else if (mb) frexp(__longlong_as_double(static_cast<long long>(mb)), &e);
  return e;
}
__device__ __forceinline__ unsigned long long oz_umax(unsigned long long a, unsigned long long b) {
  return a > b ? a : b;
}
// Balance exponent of a value of k (below): far below all others where B's row is zero or not finite, whose
// products are zero or NaN anyway.
constexpr int OZ_NO_ROW = int(0x80808080u);
__device__ __forceinline__ int oz_balance(const int* dk, int64_t k) {
  const int d = dk ? dk[k] : 0;
  return d == OZ_NO_ROW ? -(1 << 14) : d;
}
// Exponent of one entry times 2^{sign dk[k]}
__device__ __forceinline__ int oz_entry_exponent(double2 v, const int* dk, int sign, int64_t k) {
  const unsigned long long b = oz_umax(oz_abs_bits(v.x), oz_abs_bits(v.y));
  return b == 0 ? INT_MIN : (b >= 0x7FF0000000000000ull ? OZ_BAD : oz_exponent(b) + sign * oz_balance(dk, k));
}
// Power-of-two scale exponent per row of a complex128 matrix (rows x cols, ld), the max
// over Re and Im parts, with dk of the matrix whose column k is multiplied by 2^{sign dk[k]}.  One warp per row.
__global__ void oz_row_exp_kernel(const double2* __restrict__ A, int64_t rows, int64_t cols, int64_t ld,
                                  const int* __restrict__ dk, int sign, int* __restrict__ ex) {
  const int64_t row = int64_t(blockIdx.x) * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const double2* a = A + row * ld;
  if (dk) {
    int e = INT_MIN;
#pragma unroll 4
    for (int64_t k = lane; k < cols; k += 32) e = max(e, oz_entry_exponent(a[k], dk, sign, k));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) ex[row] = e == INT_MIN ? 0 : e;
    return;
  }
  unsigned long long m = 0;
#pragma unroll 4
  for (int64_t k = lane; k < cols; k += 32) {
    const double2 v = a[k];
    m = oz_umax(m, oz_umax(oz_abs_bits(v.x), oz_abs_bits(v.y)));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) m = oz_umax(m, __shfl_xor_sync(0xffffffffu, m, off));
  if (lane == 0) ex[row] = oz_exponent(m);
}
// the same per column of a matrix stored rows x cols (exponent per column, dk per row)
__global__ void oz_col_exp_kernel(const double2* __restrict__ A, int64_t rows, int64_t cols, int64_t ld,
                                  const int* __restrict__ dk, int sign, int* __restrict__ ex) {
  const int64_t col = blockIdx.x;
  __shared__ int red[8];
  int e = INT_MIN;
  if (dk) {
    for (int64_t r = threadIdx.x; r < rows; r += blockDim.x) e = max(e, oz_entry_exponent(A[r * ld + col], dk, sign, r));
  } else {
    unsigned long long m = 0;
    for (int64_t r = threadIdx.x; r < rows; r += blockDim.x) {
      const double2 v = A[r * ld + col];
      m = oz_umax(m, oz_umax(oz_abs_bits(v.x), oz_abs_bits(v.y)));
    }
    if (m) e = oz_exponent(m);
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < int(blockDim.x >> 5); ++w) e = max(e, red[w]);
    ex[col] = e == INT_MIN ? 0 : e;
  }
}
// the same for few rows (the block row of a trailing update): 32 columns x 8 lanes along the rows
__global__ void __launch_bounds__(256) oz_wide_col_exp_kernel(const double2* __restrict__ A, int64_t cols, int64_t K,
                                                              int64_t ld, const int* __restrict__ dk, int sign,
                                                              int* __restrict__ ex) {
  __shared__ int red[256];
  const int cl = threadIdx.x & 31, kl = threadIdx.x >> 5;
  const int64_t col = int64_t(blockIdx.x) * 32 + cl;
  int e = INT_MIN;
  if (col < cols) {
#pragma unroll 8
    for (int64_t k = kl; k < K; k += 8) e = max(e, oz_entry_exponent(A[k * ld + col], dk, sign, k));
  }
  red[threadIdx.x] = e;
  __syncthreads();
  if (kl == 0 && col < cols) {
    for (int w = 1; w < 8; ++w) e = max(e, red[w * 32 + cl]);
    ex[col] = e == INT_MIN ? 0 : e;
  }
}
// Products of two operands A (M x K) and B (K x N) that are both split here are balanced first: column
// k of A times, row k of B over 2^{d_k}, d_k the exponent of the largest finite entry of B's row k, for the
// trailing updates of a factorisation in the scale of the matrix' columns (col_ex).  Every k then has a
// column where B_kj attains 2^{d_k}, so the error in a row of the product is a rounding of that
// row's largest |A||B| (columns in their scale) whatever the scales of the values of k are.
// Trailing updates, CPU model with n = 400 and random matrices, componentwise backward errors of solves with
// FP64 products / digits / digits without the balance: rows scaled by 10^-8 .. 10^8 3e-15 / 3e-15 / 1e-13,
// with ten entries in half of the columns 2e-14 / 2e-14 / 2e-13, banded 4e-12 / 3e-12 / 2e-5; with d_k
// relative to the columns of the block row alone 3e-15 / 2e-13 / 3e-7.
// Products of stored factors graded by 2^-16 .. 2^16 against each other, K = 300, error over |A||B|: float-float
// 3.6e-14, digits without the balance 9e-8, with it 9e-17.
// A CTA per k (B as stored, its rows contiguous) ...
__global__ void oz_balance_kernel(const double2* __restrict__ B, int64_t N, int64_t ld, const int* __restrict__ col_ex,
                                  int* __restrict__ dk) {
  __shared__ int red[8];
  const double2* b = B + int64_t(blockIdx.x) * ld;
  int e = OZ_NO_ROW;
#pragma unroll 4
  for (int64_t j = threadIdx.x; j < N; j += blockDim.x) {
    const int v = oz_entry_exponent(b[j], nullptr, 0, 0), c = col_ex ? col_ex[j] : 0;
    if (v != INT_MIN && v != OZ_BAD) e = max(e, v - (c == OZ_NO_ROW ? 0 : c));
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < int(blockDim.x >> 5); ++w) e = max(e, red[w]);
    dk[blockIdx.x] = e;
  }
}
// ... and for a transposed B (N x K as stored): 32 values of k along the lanes, the warps share the rows
// j of a chunk, one atomic per k and CTA into dk, which starts as OZ_NO_ROW
// Both leave raw exponents; this makes them relative to the largest and leaves rows of B down to 2^-T of it
// alone (T = kFreeBinades): where rows of U are small without columns of L being large, a balance only raises
// the scales.  Forward errors of FP64 solves, EFIE matrices of 1920 unknowns, geometric means: 1.23e-14 with T = 0,
// 1.20e-14, 1.19e-14 and 1.20e-14 with 2, 3 and 5 (1.55e-14 with FP64 products); row-scaled random
// matrices n = 640, backward error 4e-15 up to 3, 6.5e-15 with 5.
constexpr int kFreeBinades = 3;
__global__ void __launch_bounds__(256) oz_balance_limit_kernel(int64_t K, int* __restrict__ dk) {
  __shared__ int red[8];
  int m = OZ_NO_ROW;
  for (int64_t k = threadIdx.x; k < K; k += 256) m = max(m, dk[k]);
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  m = red[0];
  for (int w = 1; w < 8; ++w) m = max(m, red[w]);
  for (int64_t k = threadIdx.x; k < K; k += 256) {
    const int d = dk[k];
    if (d != OZ_NO_ROW) dk[k] = min(d - m + kFreeBinades, 0);
  }
}
constexpr int64_t kBalanceRows = 512;
__global__ void __launch_bounds__(256) oz_balance_t_kernel(const double2* __restrict__ B, int64_t N, int64_t K,
                                                           int64_t ld, int* __restrict__ dk) {
  __shared__ int red[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t k = int64_t(blockIdx.x) * 32 + lane, j1 = min(N, (int64_t(blockIdx.y) + 1) * kBalanceRows);
  int e = OZ_NO_ROW;
  if (k < K) {
#pragma unroll 8
    for (int64_t j = int64_t(blockIdx.y) * kBalanceRows + warp; j < j1; j += 8) {
      const int v = oz_entry_exponent(B[j * ld + k], nullptr, 0, 0);
      if (v != INT_MIN && v != OZ_BAD) e = max(e, v);
    }
  }
  red[warp][lane] = e;
  __syncthreads();
  if (warp == 0 && k < K) {
    for (int w = 1; w < 8; ++w) e = max(e, red[w][lane]);
    if (e != OZ_NO_ROW) atomicMax(dk + k, e);
  }
}
// x 2^(55 - e) rounded to an integer (|x| < 2^e, so |F| <= 2^55), from the bit pattern:
// x = M 2^(b - 1075) with the 53-bit significand M (b the biased exponent; subnormals have
// b = 1 and no hidden bit), so F = M 2^(b - 1020 - e), a left shift of at most 2 or a right
// shift rounded to nearest (ties away from zero).  Everything below 2^-1 of the last digit
// is dropped here, the same truncation as seven successive digit roundings.
__device__ __forceinline__ long long oz_fixed(double x, int e) {
  const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
  int b = int((bits >> 52) & 0x7FF);
  unsigned long long m = bits & 0xFFFFFFFFFFFFFull;
  if (b) m |= 1ull << 52;
  else b = 1;
  const int sh = b - 1020 - e;
  unsigned long long f;
  if (sh >= 0) f = m << sh;
  else if (sh >= -60) f = (m + (1ull << (-sh - 1))) >> (-sh);
  else f = 0;
  return (bits >> 63) ? -static_cast<long long>(f) : static_cast<long long>(f);
}
// bf16 bit pattern of (byte - 128) for an integer byte in [0, 256]: the float 2^23 + byte
// minus 2^23 + 128 is exact, and a float holding an integer of magnitude <= 256 has its
// nonzero bits in the top 16
__device__ __forceinline__ uint32_t oz_bf16_bits(uint32_t byte) {
  return __float_as_uint(__uint_as_float(0x4B000000u | byte) - 8388736.0f) >> 16;
}
// Digit tiles of a matrix read as rows x K elements (element (r, k) at A[r * rs + k * ks]),
// one power-of-two exponent per row (and with dk a factor 2^{sign dk[k]} per k), zero-padded to whole tiles of TR rows x 16 k:
// tile (rt, kc, s, p) of TR x 16 bf16 at byte offset (((rt * KC + kc) * 7 + s) * 2 + p) * TR * 32.
// Z (rs = ld, ks = 1, TR = 128) and X read by columns (rs = 1, ks = ld, TR = 64) both land here.
// Digits: F = x 2^(55 - e) rounded (above) is written in balanced base 256,
// F = sum_{s=0..6} d_s 256^(6-s) with d_1..d_6 in [-128, 127] and |d_0| <= 128: adding 128 in
// each of the seven byte positions turns every digit into a plain byte (the carries of the
// balanced form are those of the addition), so d_s = byte_{6-s}(F + 0x80...80) - 128.
// A thread owns 8 consecutive k of one row, one 16-byte row of a core matrix, and writes it
// for every digit and part with one vector store; a warp covers 8 rows x 4 such groups, so
// each store instruction fills two whole 256-byte segments.
template <int TR>
__global__ void oz_split_kernel(const double2* __restrict__ A, int64_t rows, int64_t K, int64_t rs, int64_t ks,
                                bool conj, const int* __restrict__ ex, const int* __restrict__ dk, int sign, int64_t KC,
                                unsigned char* __restrict__ out) {
  constexpr int TILE = TR * OZ_KS * 2;
  constexpr unsigned long long BIAS = 0x0080808080808080ull;
  const int lane = threadIdx.x & 31;
  const int64_t row = int64_t(blockIdx.y) * 8 + (lane & 7);
  const int64_t kg = (int64_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 4 + (lane >> 3);
  if (kg >= KC * 2) return;
  const int e = row < rows ? ex[row] : 0;
  unsigned long long gr[8], gi[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int64_t k = kg * 8 + j;
    gr[j] = gi[j] = BIAS;
    if (row < rows && k < K) {
      const double2 v = A[row * rs + k * ks];
      const int ek = e - sign * oz_balance(dk, k);
      gr[j] = static_cast<unsigned long long>(oz_fixed(v.x, ek)) + BIAS;
      gi[j] = static_cast<unsigned long long>(oz_fixed(conj ? -v.y : v.y, ek)) + BIAS;
    }
  }
  const int64_t rt = row / TR, kc = kg >> 1;
  unsigned char* base = out + ((rt * KC + kc) * OZ_NT) * TILE + oz_off(int(row % TR), int(kg & 1) * 8);
#pragma unroll
  for (int s = 0; s < OZ_ND; ++s) {
    const int sh = 8 * (6 - s);
    uint32_t pr[4], pi[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      // byte 6 (digit 0) may be 256: take it with the bits above
      const uint32_t msk = s == 0 ? 0x1FFu : 0xFFu;
      pr[j] = oz_bf16_bits(uint32_t(gr[2 * j] >> sh) & msk) | (oz_bf16_bits(uint32_t(gr[2 * j + 1] >> sh) & msk) << 16);
      pi[j] = oz_bf16_bits(uint32_t(gi[2 * j] >> sh) & msk) | (oz_bf16_bits(uint32_t(gi[2 * j + 1] >> sh) & msk) << 16);
    }
    *reinterpret_cast<uint4*>(base + (s * 2 + 0) * TILE) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
    *reinterpret_cast<uint4*>(base + (s * 2 + 1) * TILE) = make_uint4(pi[0], pi[1], pi[2], pi[3]);
  }
}
constexpr int OZ_SPLIT_WARPS = 8;  // a block covers 8 rows x 8 warps x 4 groups x 8 k = 8 x 256

// ---------------------------------------------------------------- the product
// The highest order kept in each tile of 64 columns: gmax without ref.  With ref the
// operand is a correction of a matrix whose columns have the exponents ref, and what matters is
// the error against that matrix: dropping the orders above g leaves 2^{-8(g+1)} sigma tau per
// product, which is at most 2^-bits sigma 2^ref (60: 1/16 of what the product with the matrix itself
// leaves) once 8 (g + 1) >= bits - (ref - ex).  One warp per tile.
__global__ void oz_orders_kernel(const int* __restrict__ ex, const int* __restrict__ ref, int bits, int64_t N, int gmax,
                                 int* __restrict__ orders) {
  int g = ref ? 0 : gmax;
  for (int q = threadIdx.x; ref && q < OZ_TN; q += 32) {
    const int64_t c = int64_t(blockIdx.x) * OZ_TN + q;
    if (c < N) g = max(g, min(OZ_ND - 1, (bits - 1 - min(bits - 1, max(0, ref[c] - ex[c]))) / 8));
  }
  g = __reduce_max_sync(0xffffffffu, g);
  if (threadIdx.x == 0) orders[blockIdx.x] = g;
}

// The sums of one output: a = sum_g V_g 2^{unit-8g} over the orders that this leaves whole (V_g the
// order sums), added without rounding; t the others in FP32 in the same units; the value is 2^-unit (a + t).
// unit 32 (orders 0-4, the rounding of t near 2^-58 of the result) as long as K <= 2^15 keeps a
// below 2^62, 24 (orders 0-3, 2^-53) above.
__device__ __forceinline__ void oz_store(double* C, long long a, float t, int aex, int bex, int unit, double alpha,
                                         double beta) {
  const double v = double(a) + double(t);
  const double x = alpha * (aex == OZ_BAD || bex == OZ_BAD ? NAN : ldexp(v, aex + bex - 14 - unit));
  *C = beta != 0.0 ? x + beta * *C : x;
}
// One output of a piece of a tile (below).
struct OzPart {
  long long a;
  float t;
};

// One A tile with T digits of X (tiles 2 OZ_BTILE apart) into T consecutive orders, the A tile kept
// in the collector; the MMAs of a group have one instruction descriptor.
template <int T>
__device__ __forceinline__ void oz_group(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc_first,
                                         uint32_t acc_last) {
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const uint32_t acc = t == T - 1 ? acc_last : acc_first;
    const uint32_t dt = d + uint32_t(t) * OZ_TN;
    const uint64_t bt = b + uint64_t(t) * (2 * OZ_BTILE >> 4);
    if (T == 1) oz_mma_once(dt, a, bt, idesc, acc);
    else if (t == 0) oz_mma<0>(dt, a, bt, idesc, acc);
    else if (t == T - 1) oz_mma<2>(dt, a, bt, idesc, acc);
    else oz_mma<1>(dt, a, bt, idesc, acc);
  }
}

// What the MMA lane carries along.  Everything else in its inner code is a constant, so that the
// operands of the MMAs stay in uniform registers: two stages unrolled, orders and part compiled in.
struct OzMma {
  uint64_t *full, *empty;  // full by stage; empty by stage and digit of Z, digit 0 also for the digits of X
  uint32_t phase;          // phase of the full barriers, a bit per stage
  uint32_t ready;          // the next stage was seen full
  long long limit;         // polls of a wait
};
// The MMAs of one k step with the orders 0 .. G out of stage P, from digit S of Z on, part IM (0 Re,
// 1 Im).  A wait that has nothing to wait for still takes 80 cycles, and few MMAs queue up behind
// each other, so a stage has one barrier to wait for, tested before the last MMAs of the stage
// before it; its slots are given back digit by digit, which costs nothing.  `acc`: 0 where the
// step's first product into each order's accumulator (digit 0) overwrites it.
template <int G, int IM, int P, int S>
__device__ __forceinline__ void oz_step(OzMma& m, uint32_t tmem, uint32_t smem, uint32_t acc) {
  constexpr int SL = G < OZ_ND ? G : OZ_ND - 1;                    // the last digit of Z
  constexpr int T = G + 1 - S < OZ_ND ? G + 1 - S : int(OZ_ND);  // digits of X that this one meets
  if constexpr (S == (SL > 0 ? SL - 1 : 0)) m.ready = oz_test(smem_u32(&m.full[1 - P]), m.phase >> (1 - P) & 1);
  const uint64_t a = oz_desc(smem + P * OZ_STAGE + S * OZ_ASLOT), b = oz_desc(smem + P * OZ_STAGE + OZ_ND * OZ_ASLOT);
  const uint32_t d = tmem + uint32_t(S) * OZ_TN;
  // Re: Re Z Re X - Im Z Im X, Im: Re Z Im X + Im Z Re X
  // (the first product of order 7 is digit 1 of Z with digit 6 of X)
  oz_group<T>(d, a, b + uint64_t(IM * (OZ_BTILE >> 4)), oz_idesc(false), S == 0 ? acc : 1u,
              S == 0 || S + T - 1 == OZ_ND && S == 1 ? acc : 1u);
  oz_group<T>(d, a + (OZ_ATILE >> 4), b + uint64_t((1 - IM) * (OZ_BTILE >> 4)), oz_idesc(IM == 0), 1u, 1u);
  if constexpr (S > 0) oz_commit(smem_u32(&m.empty[P * OZ_ND + S]));
  if constexpr (S == SL) oz_commit(smem_u32(&m.empty[P * OZ_ND]));
  if constexpr (S < SL) oz_step<G, IM, P, S + 1>(m, tmem, smem, acc);
}
template <int G, int IM, int P>
__device__ __forceinline__ bool oz_stage(OzMma& m, uint32_t tmem, uint32_t smem, uint32_t acc) {
  if (!m.ready && !oz_wait(smem_u32(&m.full[P]), m.phase >> P & 1, m.limit)) return false;
  asm volatile("tcgen05.fence::after_thread_sync;");
  m.phase ^= 1u << P;
  oz_step<G, IM, P, 0>(m, tmem, smem, acc);
  return true;
}
// The MMAs of chunks [c0, c1) of a tile
template <int G, int IM>
__device__ __forceinline__ bool oz_tile(OzMma& m, uint32_t tmem, uint32_t smem, uint64_t* accf, uint64_t* acce, int64_t KC,
                                     int64_t c0, int64_t c1, int64_t& chunks) {
  m.ready = 0;
  for (int64_t c = c0; c < c1; ++c, ++chunks) {
    // the order accumulators are free once the flush warps have read the last chunk
    if (chunks > 0 && !oz_wait(smem_u32(acce), uint32_t((chunks - 1) & 1), m.limit)) return false;
    asm volatile("tcgen05.fence::after_thread_sync;");
    const int steps = int(std::min<int64_t>(KC - c * OZ_KCH, OZ_KCH));
    for (int k = 0; k < steps; k += 2) {  // a chunk starts at an even step
      if (!oz_stage<G, IM, 0>(m, tmem, smem, k > 0)) return false;
      if (k + 1 < steps && !oz_stage<G, IM, 1>(m, tmem, smem, 1u)) return false;
    }
    oz_commit(smem_u32(accf));
  }
  return true;
}

// The work: a tile is 128 rows x 64 columns of Re or of Im (tile index (row tile x CT + column
// tile) x 2 + part); tiles 0 .. whole - 1 whole, then the last rem = tiles - whole of them, which would
// leave most SMs without work, in `pieces` parts along k each, whose sums oz_reduce_kernel adds
// (the integers exactly, the FP32 sums in the order of k).
struct OzItem {
  int64_t tile, c0, c1;  // chunks [c0, c1) of the tile
  bool whole;
};
__device__ __forceinline__ OzItem oz_item(int64_t w, int64_t whole, int pieces, int64_t nch) {
  if (w < whole) return {w, 0, nch, true};
  const int64_t p = w - whole, q = p % pieces;
  return {whole + p / pieces, nch * q / pieces, nch * (q + 1) / pieces, pieces == 1};
}
__global__ void __launch_bounds__(OZ_THREADS, 1)
    oz_gemm_kernel(int64_t M, int64_t N, int64_t KC, const unsigned char* __restrict__ Ad,
                   const int* __restrict__ aex, const unsigned char* __restrict__ Bd, const int* __restrict__ bex,
                   const int* __restrict__ orders, int64_t whole, int pieces, int64_t items, int unit, double alpha, double beta,
                   double* __restrict__ C, int64_t ldc, OzPart* __restrict__ part, int* status) {
  extern __shared__ unsigned char oz_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(oz_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t full[2], empty[2 * OZ_ND];  // by stage; by stage and digit of Z
  __shared__ uint64_t bar_accf, bar_acce, bar_drain;
  __shared__ uint32_t tmem_sh;
  __shared__ volatile int abort_sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t CT = (N + OZ_TN - 1) / OZ_TN;
  const int64_t nch = (KC + OZ_KCH - 1) / OZ_KCH;  // chunks per tile
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_sh)),
                 "r"(OZ_TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) oz_init(smem_u32(&full[i]), OZ_ND);
    for (int i = 0; i < 2 * OZ_ND; ++i) oz_init(smem_u32(&empty[i]), 1);
    oz_init(smem_u32(&bar_accf), 1);
    oz_init(smem_u32(&bar_acce), OZ_FLUSH);
    oz_init(smem_u32(&bar_drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
    abort_sh = 0;
  }
  const long long limit = g_oz_wait_limit;
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_sh;
  auto fail = [&]() {
    abort_sh = 1;
    if (status) atomicExch(status, FOSB_ERR_TIMEOUT);
  };

  if (warp == 0) {
    // ---------------------------------------------------------- producer
    // Lane s fills digit s of Z in each stage, lane 0 also the digits of X: a wait and a copy per lane
    // and step (one lane for all took longer over them than the MMAs of the step).  Every lane
    // arrives at the stage's full barrier, those above the highest order with nothing to load.
    // The lanes meet after every step, so that none runs ahead of a barrier by more than a phase.
    const int s = lane;
    uint32_t fills0 = 0, fills1 = 0;  // of this lane's slot in each stage
    bool go = true;
    if (s < OZ_ND) {
      const uint32_t stage0 = smem_u32(smem);
      for (int64_t w = blockIdx.x; w < items && go; w += gridDim.x) {
        const OzItem item = oz_item(w, whole, pieces, nch);
        const int64_t rt = item.tile / (2 * CT), ct = item.tile / 2 % CT;
        const int G = orders[ct];
        const int64_t k1 = std::min<int64_t>(KC, item.c1 * OZ_KCH);
        // the digits up to the highest order are the first tiles of each operand's step
        const uint32_t bbytes = s == 0 ? uint32_t(min(G + 1, int(OZ_ND))) * 2 * OZ_BTILE : 0u;
        for (int64_t kc = item.c0 * OZ_KCH; kc < k1 && go; ++kc) {  // (starts even)
          const int p = int(kc & 1);
          const uint32_t turn = p ? fills1 : fills0;
          bool ok = !abort_sh;
          if (ok && s <= G && turn > 0 && !oz_wait(smem_u32(&empty[p * OZ_ND + s]), (turn - 1) & 1, limit)) {
            fail();
            ok = false;
          }
          go = __all_sync((1u << OZ_ND) - 1u, ok);
          if (!go) break;
          const uint32_t bar = smem_u32(&full[p]), dst = stage0 + p * OZ_STAGE;
          oz_expect_tx(bar, s <= G ? OZ_ASLOT + bbytes : 0u);
          if (s <= G) {
            (p ? fills1 : fills0) = turn + 1;
            if (s == 0) oz_bulk_load(dst + OZ_ND * OZ_ASLOT, Bd + (ct * KC + kc) * OZ_BSLOT, bbytes, bar);
            oz_bulk_load(dst + s * OZ_ASLOT, Ad + (rt * KC + kc) * (OZ_NT * OZ_ATILE) + s * OZ_ASLOT, OZ_ASLOT, bar);
          }
        }
      }
      // no copy may land after the kernel has left (it can leave early where a wait gave up); lane 0
      // has filled its slot in every step
      if (s == 0 && fills0 > 0) oz_wait(smem_u32(&full[0]), (fills0 - 1) & 1);
      if (s == 0 && fills1 > 0) oz_wait(smem_u32(&full[1]), (fills1 - 1) & 1);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------------------- MMA issuer
    if (oz_elect()) {
      OzMma m = {full, empty, 0u, 0u, limit};
      const uint32_t stage0 = smem_u32(smem);
      int64_t chunks = 0;
      for (int64_t w = blockIdx.x; w < items && !abort_sh; w += gridDim.x) {
        const OzItem item = oz_item(w, whole, pieces, nch);
        auto run = [&](auto g) {
          constexpr int G = decltype(g)::value;
          return item.tile & 1 ? oz_tile<G, 1>(m, tmem, stage0, &bar_accf, &bar_acce, KC, item.c0, item.c1, chunks)
                               : oz_tile<G, 0>(m, tmem, stage0, &bar_accf, &bar_acce, KC, item.c0, item.c1, chunks);
        };
        bool ok;
        switch (orders[item.tile / 2 % CT]) {
          case 0: ok = run(std::integral_constant<int, 0>()); break;
          case 1: ok = run(std::integral_constant<int, 1>()); break;
          case 2: ok = run(std::integral_constant<int, 2>()); break;
          case 3: ok = run(std::integral_constant<int, 3>()); break;
          case 4: ok = run(std::integral_constant<int, 4>()); break;
          case 5: ok = run(std::integral_constant<int, 5>()); break;
          case 6: ok = run(std::integral_constant<int, 6>()); break;
          default: ok = run(std::integral_constant<int, 7>()); break;
        }
        if (!ok) {
          fail();
          break;
        }
      }
      oz_commit(smem_u32(&bar_drain));  // completes once every MMA above has finished
      if (!oz_wait(smem_u32(&bar_drain), 0u)) fail();
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------- flush and epilogue (warps 2-9)
    // TMEM lane group warp % 4 (rows), column half (warp - 2) / 4 of the tile
    const int lane_base = (warp & 3) * 32;
    const int c0 = ((warp - 2) >> 2) * OZ_HN;
    const int r_local = lane_base + lane;
    const uint32_t tbase = tmem + (uint32_t(lane_base) << 16) + uint32_t(c0);
    int64_t chunks = 0;
    bool stopped = false;
    for (int64_t w = blockIdx.x; w < items; w += gridDim.x) {
      const OzItem item = oz_item(w, whole, pieces, nch);
      const int64_t rt = item.tile / (2 * CT), ct = item.tile / 2 % CT;
      const int G = orders[ct];
      long long a[OZ_HN];
      float t[OZ_HN];
#pragma unroll
      for (int j = 0; j < OZ_HN; ++j) {
        a[j] = 0ll;
        t[j] = 0.f;
      }
      for (int64_t c = item.c0; c < item.c1 && !stopped; ++c, ++chunks) {
        const bool full_in_time = oz_wait<true>(smem_u32(&bar_accf), uint32_t(chunks & 1), limit);
        if (!full_in_time) fail();
        // the stop decision is the same in all eight warps: the barrier itself hands out the OR (a flag
        // read behind it could already be the next chunk's)
        stopped = oz_any(!full_in_time);
        if (stopped) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        // eight columns of two orders at a time, the next ones on their way during the arithmetic
        uint32_t v[2][8], u[2][8];
        auto load = [&](int g, int j0, int buf) {  // orders g and g + 1
          oz_ld8(tbase + uint32_t(g * OZ_TN + j0), v[buf]);
          if (g + 1 <= G) oz_ld8(tbase + uint32_t((g + 1) * OZ_TN + j0), u[buf]);
        };
        auto digit = [](uint32_t x) { return __float2int_rn(__uint_as_float(x)); };
        const float w5 = unit == 32 ? 0x1p-8f : 0x1p-16f;  // 2^{unit-40}
        load(0, 0, 0);
#pragma unroll
        for (int g = 0; g <= OZ_ND; g += 2) {
          if (g > G) break;
#pragma unroll
          for (int j0 = 0; j0 < OZ_HN; j0 += 8) {
            const int buf = j0 >> 3 & 1;
            oz_wait_ld(v[buf], u[buf]);
            if (j0 + 8 < OZ_HN) load(g, j0 + 8, 1 - buf);
            else if (g + 2 <= G) load(g + 2, 0, 0);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float x = __uint_as_float(v[buf][j]), y = __uint_as_float(u[buf][j]);
              if (g == 0)  // V_0 2^8 + V_1 fits 32 bits (|V_0| <= 2^22, |V_1| <= 2^23)
                a[j0 + j] += (long long)(digit(v[buf][j]) * 256 + (G >= 1 ? digit(u[buf][j]) : 0)) * (1 << (unit - 8));
              else if (g == 2)
                a[j0 + j] += (long long)digit(v[buf][j]) * (1 << (unit - 16)) +
                             (G >= 3 ? (long long)digit(u[buf][j]) * (1 << (unit - 24)) : 0ll);
              else if (g == 4) {
                if (unit == 32) a[j0 + j] += digit(v[buf][j]);
                else t[j0 + j] = fmaf(x, 0x1p-8f, t[j0 + j]);
                if (G >= 5) t[j0 + j] = fmaf(y, w5, t[j0 + j]);
              } else {
                if (G >= 7) t[j0 + j] = fmaf(y, w5 * 0x1p-16f, t[j0 + j]);
                t[j0 + j] = fmaf(x, w5 * 0x1p-8f, t[j0 + j]);
              }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        oz_arrive(smem_u32(&bar_acce));
      }
      if (stopped) {  // what a wait that gave up leaves undone becomes NaN
#pragma unroll
        for (int j = 0; j < OZ_HN; ++j) t[j] = NAN;
      }
      const int64_t row = rt * OZ_TM + r_local;
      if (!item.whole) {
        OzPart* p = part + ((w - whole) * OZ_TM + r_local) * OZ_TN + c0;
#pragma unroll
        for (int j = 0; j < OZ_HN; ++j) p[j] = {a[j], t[j]};
      } else if (row < M) {
        const int ae = aex[row];
#pragma unroll
        for (int j = 0; j < OZ_HN; ++j) {
          const int64_t col = ct * OZ_TN + c0 + j;
          if (col < N) oz_store(C + (row * ldc + col) * 2 + (item.tile & 1), a[j], t[j], ae, bex[col], unit, alpha, beta);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM_COLS));
}

__global__ void oz_reduce_kernel(int64_t M, int64_t N, int64_t whole, int pieces, const OzPart* __restrict__ part,
                                 const int* __restrict__ aex, const int* __restrict__ bex, int unit, double alpha,
                                 double beta, double* __restrict__ C, int64_t ldc) {
  const int64_t CT = (N + OZ_TN - 1) / OZ_TN, tile = whole + blockIdx.x;
  const int e = int(blockIdx.y) * 256 + int(threadIdx.x);  // element of the tile
  const int64_t row = tile / (2 * CT) * OZ_TM + e / OZ_TN, col = tile / 2 % CT * OZ_TN + e % OZ_TN;
  if (row >= M || col >= N) return;
  OzPart s = {0, 0.f};
  for (int q = 0; q < pieces; ++q) {
    const OzPart p = part[(int64_t(blockIdx.x) * pieces + q) * (OZ_TM * OZ_TN) + e];
    s.a += p.a;
    s.t += p.t;
  }
  oz_store(C + (row * ldc + col) * 2 + (tile & 1), s.a, s.t, aex[row], bex[col], unit, alpha, beta);
}

inline unsigned oz_cdiv(int64_t a, int64_t b) { return unsigned((a + b - 1) / b); }

}  // namespace

size_t oz_a_bytes(int64_t M, int64_t K) {
  return size_t((M + OZ_TM - 1) / OZ_TM) * size_t((K + OZ_KS - 1) / OZ_KS) * OZ_NT * OZ_ATILE;
}

// Exponents (of the rows, times 2^{sign dk[k]} with dk) of a matrix read as rows x K
static void oz_exponents(const double2* X, int64_t rows, int64_t K, int64_t rs, int64_t ks, const int* dk, int sign,
                         int* ex, cudaStream_t s) {
  if (ks == 1) oz_row_exp_kernel<<<oz_cdiv(rows, 8), 256, 0, s>>>(X, rows, K, rs, dk, sign, ex);
  else if (K < 128) oz_wide_col_exp_kernel<<<oz_cdiv(rows, 32), 256, 0, s>>>(X, rows, K, ks, dk, sign, ex);
  else oz_col_exp_kernel<<<unsigned(rows), 256, 0, s>>>(X, K, rows, ks, dk, sign, ex);
}
// Digit tiles of a matrix read as rows x K with the exponents ex of its rows, in tiles of TR rows; with dk
// balanced, as the left (sign +1) or the right (sign -1) operand
template <int TR>
static cudaError_t oz_digits(const double2* X, int64_t rows, int64_t K, int64_t rs, int64_t ks, bool conj,
                             const int* dk, int sign, const int* ex, void* digits, cudaStream_t s) {
  const int64_t KC = (K + OZ_KS - 1) / OZ_KS, RP = (rows + TR - 1) / TR * TR;
  if (RP / 8 > 65535) return cudaErrorInvalidValue;
  oz_split_kernel<TR><<<dim3(oz_cdiv(KC * 2, OZ_SPLIT_WARPS * 4), unsigned(RP / 8)), OZ_SPLIT_WARPS * 32, 0, s>>>(
      X, rows, K, rs, ks, conj, ex, dk, sign, KC, static_cast<unsigned char*>(digits));
  return launched(1);
}

cudaError_t oz_prepare_a(const void* A, int64_t M, int64_t K, int64_t lda, void* digits, int* ex, cudaStream_t s) {
  if (M <= 0 || K <= 0) return cudaSuccess;
  ProfScope prof("oz_prep", s, 44.0 * double(M) * double(K));  // bytes read + written
  const double2* a = static_cast<const double2*>(A);
  oz_exponents(a, M, K, lda, 1, nullptr, 0, ex, s);
  note_launches(1);
  return oz_digits<OZ_TM>(a, M, K, lda, 1, false, nullptr, 0, ex, digits, s);
}

// Digit tiles and orders of an N-column right operand
static size_t oz_right_bytes(int64_t N, int64_t K) {
  return size_t((N + OZ_TN - 1) / OZ_TN) * (size_t((K + OZ_KS - 1) / OZ_KS) * OZ_BSLOT + sizeof(int));
}

// b_ex: the exponents of op(B)'s columns; right: oz_right_bytes(N, K) of scratch, or null to allocate
static cudaError_t oz_product(int opB, int64_t M, int64_t N, int64_t K, double alpha, const void* a_digits,
                              const int* a_ex, const void* B, int64_t ldb, double beta, void* C, int64_t ldc,
                              const int* b_ex, const int* ref_ex, int bits, const int* dk, int gmax, int* status,
                              void* right, cudaStream_t s) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  static bool attr[64] = {};
  static int nsm[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr[dev]) {
    cudaError_t e = cudaFuncSetAttribute(oz_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&nsm[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    attr[dev] = true;
  }
  const int64_t KC = (K + OZ_KS - 1) / OZ_KS, CT = (N + OZ_TN - 1) / OZ_TN, nch = (KC + OZ_KCH - 1) / OZ_KCH;
  if (CT * OZ_TN / 8 > 65535) return cudaErrorInvalidValue;
  // the tiles that would not fill the chip, in as many pieces of at least 8 chunks as there are SMs for
  const int64_t sms = std::max(nsm[dev], 1), tiles = ((M + OZ_TM - 1) / OZ_TM) * CT * 2, rem = tiles % sms;
  const int64_t whole = tiles - rem;
  const int pieces = rem ? int(std::max<int64_t>(1, std::min<int64_t>(sms / rem, nch / 8))) : 1;
  const int64_t items = whole + rem * pieces;
  const int unit = K <= (1 << 15) ? 32 : 24;  // of the integer sums (oz_store)
  // the pieces' sums, then digit tiles of B, then the orders
  const size_t bbytes = size_t(CT) * size_t(KC) * OZ_BSLOT;
  const size_t pbytes = pieces > 1 ? sizeof(OzPart) * size_t(rem * pieces) * OZ_TM * OZ_TN : 0;
  Scratch own(s);
  if (!right || pieces > 1) {
    const cudaError_t e = own.alloc(pbytes + oz_right_bytes(N, K));
    if (e != cudaSuccess) return e;
    right = static_cast<char*>(own.p) + pbytes;
  }
  OzPart* part = static_cast<OzPart*>(own.p);
  unsigned char* bd = static_cast<unsigned char*>(right);
  int* orders = reinterpret_cast<int*>(bd + bbytes);
  cudaError_t e = oz_digits<OZ_TN>(static_cast<const double2*>(B), N, K, opB == OP_N ? 1 : ldb, opB == OP_N ? ldb : 1, opB == OP_C,
                       dk, -1, b_ex, bd, s);
  if (e != cudaSuccess) return e;
  oz_orders_kernel<<<unsigned(CT), 32, 0, s>>>(b_ex, ref_ex, bits, N, gmax, orders);
  {
    ProfScope prof("gemm_oz", s, 8.0 * double(M) * double(N) * double(K));
    oz_gemm_kernel<<<unsigned(std::min(items, sms)), OZ_THREADS, OZ_SMEM, s>>>(
        M, N, KC, static_cast<const unsigned char*>(a_digits), a_ex, bd, b_ex, orders, whole, pieces, items, unit, alpha, beta,
        static_cast<double*>(C), ldc, part, status);
    if (pieces > 1)
      oz_reduce_kernel<<<dim3(unsigned(rem), OZ_TM * OZ_TN / 256), 256, 0, s>>>(
          M, N, whole, pieces, part, a_ex, b_ex, unit, alpha, beta, static_cast<double*>(C), ldc);
  }
  return launched(pieces > 1 ? 3 : 2);
}

cudaError_t oz_gemm(int64_t M, int64_t N, int64_t K, double alpha, const void* a_digits, const int* a_ex,
                    const void* B, int64_t ldb, double beta, void* C, int64_t ldc, int* b_ex, const int* ref_ex,
                    int bits, int* status, cudaStream_t s) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  oz_exponents(static_cast<const double2*>(B), N, K, 1, ldb, nullptr, 0, b_ex, s);
  note_launches(1);
  return oz_product(OP_N, M, N, K, alpha, a_digits, a_ex, B, ldb, beta, C, ldc, b_ex, ref_ex, bits, nullptr, OZ_ND - 1, status,
                    nullptr, s);
}

// All the memory of a balanced product that is not cut into pieces along k (K <= 64 is one chunk)
size_t oz_balanced_bytes(int64_t M, int64_t N, int64_t K) {
  return oz_a_bytes(M, K) + (oz_right_bytes(N, K) + 15) / 16 * 16 + sizeof(int) * size_t(M + N + K);
}

// C <- beta C + alpha op(A) op(B), balanced along k, with the digit orders up to gmax; scratch:
// oz_balanced_bytes(M, N, K)
static cudaError_t oz_balanced(int opA, int opB, int64_t M, int64_t N, int64_t K, double alpha, const void* A,
                               int64_t lda, const void* B, int64_t ldb, double beta, void* C, int64_t ldc,
                               const int* col_ex, void* scratch, int gmax, int* status, cudaStream_t s) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  char* dig = static_cast<char*>(scratch);
  char* right = dig + oz_a_bytes(M, K);
  int* dk = reinterpret_cast<int*>(right + (oz_right_bytes(N, K) + 15) / 16 * 16);
  int *a_ex = dk + K, *b_ex = a_ex + M;
  const double2 *a = static_cast<const double2*>(A), *b = static_cast<const double2*>(B);
  if (opB == OP_N) {
    oz_balance_kernel<<<unsigned(K), 256, 0, s>>>(b, N, ldb, col_ex, dk);
  } else {
    const cudaError_t e = cudaMemsetAsync(dk, 0x80, sizeof(int) * size_t(K), s);
    if (e != cudaSuccess) return e;
    oz_balance_t_kernel<<<dim3(oz_cdiv(K, 32), oz_cdiv(N, kBalanceRows)), 256, 0, s>>>(b, N, K, ldb, dk);
  }
  oz_balance_limit_kernel<<<1, 256, 0, s>>>(K, dk);
  const int64_t rs = opA == OP_N ? lda : 1, ks = opA == OP_N ? 1 : lda;
  oz_exponents(a, M, K, rs, ks, dk, 1, a_ex, s);
  oz_exponents(b, N, K, opB == OP_N ? 1 : ldb, opB == OP_N ? ldb : 1, dk, -1, b_ex, s);
  note_launches(4);
  const cudaError_t e = oz_digits<OZ_TM>(a, M, K, rs, ks, opA == OP_C, dk, 1, a_ex, dig, s);
  if (e != cudaSuccess) return e;
  return oz_product(opB, M, N, K, alpha, dig, a_ex, B, ldb, beta, C, ldc, b_ex, nullptr, 0, dk, gmax, status, right, s);
}

cudaError_t oz_update(int64_t M, int64_t N, int64_t K, const void* L, int64_t ldl, const void* U, int64_t ldu, void* C,
                      int64_t ldc, const int* col_ex, void* scratch, int* status, cudaStream_t s) {
  return oz_balanced(OP_N, OP_N, M, N, K, -1.0, L, ldl, U, ldu, 1.0, C, ldc, col_ex, scratch, OZ_ND, status, s);
}

cudaError_t DigitStatus::get(int** p) {
  if (!word_.p) {
    cudaError_t e = word_.alloc(sizeof(int));
    if (e == cudaSuccess) e = cudaMemsetAsync(word_.p, 0, sizeof(int), word_.s);
    if (e != cudaSuccess) return e;
  }
  *p = word_.as<int>();
  return cudaSuccess;
}

fosb_status DigitStatus::check(const char* call) {
  if (!word_.p) return FOSB_OK;
  int status = 0;
  FOSB_CUDA(cudaMemcpyAsync(&status, word_.p, sizeof(int), cudaMemcpyDeviceToHost, word_.s));
  // (polled: a synchronisation would also give the pool's free memory back, which the next call maps again)
  cudaError_t e;
  while ((e = cudaStreamQuery(word_.s)) == cudaErrorNotReady) std::this_thread::yield();
  FOSB_CUDA(e);
  if (status == FOSB_ERR_TIMEOUT) return fail(FOSB_ERR_TIMEOUT, std::string(call) + ": tensor-core wait timed out");
  return FOSB_OK;
}

// FP64-class op(A) op(B) for any operands: digits of both, made here.  The digit path takes over at
// K = 128: below, the passes over the outputs are most of either (digits / float-float, us: 1000 x
// 1000 x 64 158 / 164, 3000 x 3000 x 32 707 / 650, 1000 x 1000 x 16 148 / 72), above it wins at any
// M and N (100 x 16 x 100 91 / 131, 3 x 500 x 7503 630 / 653, 500 x 500 x 500 168 / 559, 7503 x 363
// x 1089 980 / 5708, 7503 x 7503 x 642 9685 / 61614).
cudaError_t gemm_c128_fp64class(int opA, int opB, int64_t M, int64_t N, int64_t K, double alpha, const void* A,
                                int64_t lda, const void* B, int64_t ldb, double beta, void* C, int64_t ldc,
                                DigitStatus& st, cudaStream_t s) {
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) cudaGetLastError();
  if (M > 0 && N > 8 && K >= 128 && M <= 65535 * 8 - 128 &&
      N <= 65535 * 8 - 64 && capture == cudaStreamCaptureStatusNone) {
    void* d = nullptr;
    int* status = nullptr;
    cudaError_t e = st.get(&status);
    if (e == cudaSuccess) e = device_alloc(&d, oz_balanced_bytes(M, N, K), s);
    if (e == cudaSuccess)
      e = oz_balanced(opA, opB, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, nullptr, d, OZ_ND - 1, status, s);
    if (d) cudaFreeAsync(d, s);
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();  // no room for the digits (28 bytes per entry): float-float needs 16
  }
  return gemm_c128_ff(opA, opB, M, N, K, alpha, 0.0, A, lda, B, ldb, beta, C, ldc, s);
}

}  // namespace fosb

// Sets the poll limit of the digit kernel's waits on the current device (polls <= 0: the default).
cudaError_t fosb::set_wait_limit_digits(long long polls) {
  const long long v = polls > 0 ? polls : kOzSpinLimit;
  return cudaMemcpyToSymbol(g_oz_wait_limit, &v, sizeof(v));
}

extern "C" fosb_status fosb_zgemm_fp64class(int64_t M, int64_t N, int64_t K, const void* A, int64_t lda, const void* B,
                                            int64_t ldb, void* C, int64_t ldc, int method, void* stream) {
  using namespace fosb;
  if (M < 0 || N < 0 || K < 0 || (M > 0 && N > 0 && (!A || !B || !C)) || lda < K || ldb < N || ldc < N)
    return fail(FOSB_ERR_INVALID_ARG, "fosb_zgemm_fp64class: bad arguments");
  if (method != 0 && method != 1) return fail(FOSB_ERR_INVALID_ARG, "fosb_zgemm_fp64class: method must be 0 or 1");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (M == 0 || N == 0) return FOSB_OK;
  if (K == 0) {
    FOSB_CUDA(cudaMemset2DAsync(C, ldc * 16, 0, N * 16, M, s));
    return FOSB_OK;
  }
  if (method == 1) {
    FOSB_CUDA(gemm_c128_ff(OP_N, OP_N, M, N, K, 1.0, 0.0, A, lda, B, ldb, 0.0, C, ldc, s));
    return FOSB_OK;
  }
  Scratch dig(s), ex(s);
  DigitStatus st(s);
  int* status = nullptr;
  FOSB_CUDA(dig.alloc(oz_a_bytes(M, K)));
  FOSB_CUDA(ex.alloc(sizeof(int) * size_t(M + N)));
  FOSB_CUDA(st.get(&status));
  FOSB_CUDA(oz_prepare_a(A, M, K, lda, dig.p, ex.as<int>(), s));
  FOSB_CUDA(oz_gemm(M, N, K, 1.0, dig.p, ex.as<int>(), B, ldb, 0.0, C, ldc, ex.as<int>() + M, nullptr, 0,
                    status, s));
  return st.check("fosb_zgemm_fp64class");
}

