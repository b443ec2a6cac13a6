// Trailing update C -= A B of the blocked complex64 LU on the tcgen05 tensor cores, fed by
// bulk copies of operands split once per block into two fp16 values per real number.
//
// The split.  A and B are first balanced along k: row k of B over 2^{d_k}, column k of A times 2^{d_k},
// d_k the exponent of the largest entry of B's row k in the scale of the matrix' columns.  Then every row
// i of A and column j of B is scaled by a power of two that brings its largest |Re|, |Im| into
// [2^14, 2^15), and x s = x_h + x_l with x_h = fp16(x s), x_l = fp16(x s - x_h):
//   x y ~ x_h y_h + x_h y_l + x_l y_h,
// accumulated in FP32 and scaled back exactly.  fp16 carries 11 significand bits as TF32 does, so
// the pair holds 22 bits like the 3xTF32 split (down to 2^-18 of the row's largest value, below
// that the error is 2^-40 of it), and one MMA covers 16 values of k instead of 8: half the tensor time.
// Error against 64 bits at K = 256, normwise: 1.9e-6 (3xTF32 3.6e-6) on uniform operands, on operands graded
// over six decades inside their rows and on ones scaled by row and column over as many: half as
// many accumulations in the tensor core.
// The balance is for matrices whose rows differ in scale: U12's rows then carry the scales and L21's
// columns their inverses, so the products are of one size but lie far below a row's times a column's
// largest value.  With it a row's error is below 2^-40 of the largest |L||U| in that row, columns taken
// in the matrix' own scale (every k has a column where U_kj attains 2^{d_k}), as far as a single value
// is below the 22 bits: CPU model, K = 256, n = 400, scaled, banded and sparse matrices, factor error over
// |L||U| as with 3xTF32 (1e-7), 3e-4 without the balance; matrices of blocks with scales of their own
// are normwise in each row only (4e-5 of |L||U|; backward errors of solves as with 3xTF32).
//
// Split once, copied many times.  A (L21, M x K) and B (U12, K x N) are each split by one
// pass per column block (K <= 256) into the exact shared-memory image the MMAs read: for every
// 128-row (or 128-column) tile and 16-wide k-slab, 4 KB "parts" in the canonical no-swizzle
// K-major layout (8-row x 16-byte core matrices; 128 B between the two core matrices of a
// slab, 256 B between 8-row groups).  Per slab, A has 4 parts (Re_h, Re_l, Im_h, Im_l) and
// B has 6: high [Br_h | Bi_h | -Br_h] then low [Br_l | Bi_l | -Br_l].  A tile's stage is
// then two plain cp.async.bulk copies (16 KB + 24 KB): no per-CTA split, no scattered
// shared-memory stores, and a 3-deep ring that hides the L2 latency.
//
// Complex product with N = 256 MMAs.  The accumulator holds [Re | Im] of a 128 x 128 complex
// tile in 256 TMEM columns, and B is read through two 256-row windows of the contiguous
// parts:  [Br | Bi] (at Br) and [Bi | -Br] (at Bi), so
//   D += A_r [Br | Bi] + (-A_i) [Bi | -Br] = [Ar Br - Ai Bi | Ar Bi + Ai Br]
// (the -A_i by the instruction's negate-A bit): 6 MMAs of 128 x 256 x 16 per slab instead of
// 12 of 128 x 128 x 16, with half the B-operand reads per useful flop.
//
// Roles (persistent, one CTA per SM, tiles in super-rows of 16 row tiles for L2 reuse):
//   warp 0  producer: per slab waits empty[s], expect_tx 40 KB, two bulk copies;
//   warp 1  MMA issuer: waits full[s], 6 MMAs into accumulator buffer b, commits empty[s];
//           after a tile's last slab commits tfull[b];
//   warps 2-9 epilogue, two groups of four (TMEM lane quarters 2, 3, 0, 1): per 32-column quarter,
//           C is prefetched by cp.async into a padded shared tile, the accumulator row of each thread
//           is subtracted in place, and the quarter is stored with coalesced 16-byte writes.
// The 59 updates of an N = 15360 factorisation: 26.4 ms with one group on 64-column halves, 22.4 ms so.
// What bounds it: operands and C reach the SMs at 11 TB/s, and the MMAs' operand reads with the copies'
// writes want 146 of the 128 B a clock that shared memory gives at the full MMA rate (an elected MMA
// lane and waits tested ahead changed nothing).
// Every wait is bounded; a time-out sets the status word and an abort flag, the MMA thread
// drains its MMAs and the producer waits for its copies in flight before TMEM is freed.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "fosb_internal.h"

namespace fosb {
namespace {

constexpr int U_TM = 128, U_TN = 128;          // tile: 128 rows x 128 complex columns
constexpr int U_KB = kLuBlock;                 // largest k extent of a split block (16 slabs)
constexpr int U_KS = 16;                       // k values per slab
constexpr int U_SLABS = U_KB / U_KS;
constexpr int U_PART = 4096;                   // one 128 x 16 fp16 part
constexpr int U_ABYTES = 4 * U_PART;           // A parts of one slab
constexpr int U_BBYTES = 6 * U_PART;           // B parts of one slab
constexpr int U_STAGE = U_ABYTES + U_BBYTES;   // 40 KB
constexpr int U_STAGES = 3;
constexpr int U_EPI_N = 32;                    // columns of C that an epilogue group holds at a time
constexpr int U_EPI_LD = U_EPI_N + 2;          // padded float2 row of them (16-byte rows)
constexpr int U_EPI_BYTES = 2 * U_TM * U_EPI_LD * 8;
constexpr int U_EPI_OFF = U_STAGES * U_STAGE;
constexpr int U_SMEM = U_EPI_OFF + U_EPI_BYTES + 1024;  // + alignment slack
constexpr int U_THREADS = 10 * 32;              // producer, MMA, two epilogue groups of four warps
constexpr int U_GROUP = 16;                    // row tiles per super-row
constexpr long long U_SPIN = 1ll << 24;
static_assert(U_SMEM <= 227 * 1024, "stages and drain tile exceed shared memory");

__device__ __forceinline__ uint32_t su32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
// byte offset of element (row, k), k < 16, of a part: 8-row groups 256 B apart, k halves 128 B apart
__host__ __device__ __forceinline__ int part_off(int row, int k) {
  return (row >> 3) * 256 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}
__device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
  return uint64_t((addr >> 4) & 0x3FFF) | (uint64_t(128 >> 4) << 16) | (uint64_t(256 >> 4) << 32) |
         (uint64_t(1) << 46);
}
// kind::f16: D f32 (bits 4-5 = 1), A and B fp16 (bits 7-9, 10-12 = 0), K-major, N = 256, M = 128,
// optional negate-A (bit 13)
__host__ __device__ constexpr uint32_t u_idesc(bool neg_a) {
  return (1u << 4) | (neg_a ? (1u << 13) : 0u) | (uint32_t(256 >> 3) << 17) | (uint32_t(U_TM >> 4) << 24);
}
__device__ __forceinline__ void u_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ bool u_wait(uint32_t mbar, uint32_t parity) {
  for (long long i = 0; i < U_SPIN; ++i) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity));
    if (done) return true;
    __nanosleep(32);
  }
  return false;
}
__device__ __forceinline__ void u_init(uint32_t a, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(n));
}
__device__ __forceinline__ void u_arrive(uint32_t a) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(a));
}
__device__ __forceinline__ void u_expect_tx(uint32_t a, uint32_t bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(a), "r"(bytes));
}
__device__ __forceinline__ void u_bulk(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(mbar)
               : "memory");
}
__device__ __forceinline__ void u_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar));
}
__device__ __forceinline__ void u_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
}
__device__ __forceinline__ void u_bar(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n)); }
// 16-byte global -> shared copy that bypasses the registers; bytes < 16 zero-fills the rest
__device__ __forceinline__ void u_cp16(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
// float2 index of the 16-byte piece holding columns (2 j, 2 j + 1) of row r in a 32-column
// buffer; the 272-byte row pitch keeps 8 consecutive rows reading piece j in 8 different
// bank groups (row-per-thread phase) and a row's 16 pieces contiguous (coalesced phases)
__device__ __forceinline__ int u_piece(int r, int j) { return r * U_EPI_LD + (j << 1); }
__device__ __forceinline__ void u_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void u_cp_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// ---------------------------------------------------------------- splits
// 2^e for a normal result, and x 2^e for |e| <= 252 as two exact factors
__device__ __forceinline__ float pow2(int e) { return __uint_as_float(unsigned(127 + e) << 23); }
__device__ __forceinline__ float scale2(float x, int e) { return x * pow2(e >> 1) * pow2(e - (e >> 1)); }
// Biased exponent of the larger of |Re|, |Im|: kNone for zero, kBad for infinities and NaN.
constexpr int kNone = -(1 << 20), kBad = 1 << 20;
__device__ __forceinline__ int value_exp(float2 v) {
  const unsigned b = max(__float_as_uint(v.x) & 0x7FFFFFFFu, __float_as_uint(v.y) & 0x7FFFFFFFu);
  return b == 0u ? kNone : (b >= 0x7F800000u ? kBad : int(b >> 23));
}
// Exponent of the power of two that brings a row's or column's largest |Re|, |Im| (biased exponent e)
// into [2^14, 2^15), as far as it and its inverse are normal floats; 0 for zero and for what is not finite.
__device__ __forceinline__ int scale_exp(int e) {
  return e <= kNone / 2 || e >= kBad / 2 ? 0 : max(-126, min(126, 14 + 127 - e));
}
// fp16 pair of 8 scaled values, packed for two 16-byte stores
__device__ __forceinline__ void split8(const float (&x)[8], uint4& hi, uint4& lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float a = x[2 * i], b = x[2 * i + 1];
    const __half2 hh = __floats2half2_rn(a, b);
    const float2 back = __half22float2(hh);
    const __half2 ll = __floats2half2_rn(a - back.x, b - back.y);
    h[i] = *reinterpret_cast<const uint32_t*>(&hh);
    l[i] = *reinterpret_cast<const uint32_t*>(&ll);
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}
__device__ __forceinline__ uint4 neg8(uint4 v) {
  return make_uint4(v.x ^ 0x80008000u, v.y ^ 0x80008000u, v.z ^ 0x80008000u, v.w ^ 0x80008000u);
}

// dk[k] = the largest value_exp of B's row k less that of its column (col_ex), over the finite entries; kNone for
// a zero row and k >= K.  A CTA per k.  Bound by latency: 6 us per update of an
// N = 15360 factorisation; all 59 updates with their splits 24.9 ms, 24.3 ms without the balance.
__global__ void __launch_bounds__(512) row_balance_kernel(int64_t N, int K, const float2* __restrict__ B, int64_t ldb,
                                                          const int* __restrict__ col_ex, int* __restrict__ dk) {
  __shared__ int red[16];
  const int k = int(blockIdx.x);
  int d = kNone;
  if (k < K) {
    const float2* b = B + int64_t(k) * ldb;
#pragma unroll 8
    for (int64_t j = threadIdx.x; j < N; j += 512) {
      const int e = value_exp(b[j]), c = col_ex[j];
      if (e != kNone && e != kBad) d = max(d, e - (c < kNone ? 0 : c));  // (none: a column without finite values)
    }
  }
  d = __reduce_max_sync(0xffffffffu, d);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = d;
  __syncthreads();
  if (threadIdx.x >= 32) return;
  d = __reduce_max_sync(0xffffffffu, red[threadIdx.x & 15]);
  if (threadIdx.x == 0) dk[k] = d;
}
// The largest of the balance exponents, by a warp.  The balance in use is relative to it: rows of B down to
// 2^-kFreeBinades of the largest are left alone (the split carries them, and where rows of U are small without
// columns of L being large a balance only raises the scales), and none is below -100 so that the scales
// stay normal floats (zero rows have that too, their products are zero).
constexpr int kFreeBinades = 8;
__device__ __forceinline__ int balance_max(const int* __restrict__ dk, int lane) {
  int d = kNone;
#pragma unroll
  for (int i = 0; i < U_KB; i += 32) d = max(d, dk[i + lane]);
  return __reduce_max_sync(0xffffffffu, d);
}
// The balance exponents of 8 values of k from k0 on (a multiple of 8)
__device__ __forceinline__ void balance8(const int* __restrict__ dk, int k0, int dmax, int (&d)[8]) {
  const int4 p = *reinterpret_cast<const int4*>(dk + k0), q = *reinterpret_cast<const int4*>(dk + k0 + 4);
  const int v[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
  for (int i = 0; i < 8; ++i) d[i] = max(min(v[i] - dmax + kFreeBinades, 0), -100);
}

// A (M x K, lda), K <= 256 in nslab = ceil(K / 16) slabs: out[(rt * nslab + s) * 16 KB + p * 4 KB +
// part_off(r, k)], parts Re_h, Re_l, Im_h, Im_l; zero outside M x K; inv[row] the inverse scales.  A warp per
// 8 rows: lane (row, group) takes every fourth group of 8 values of k, first for the row's largest
// balanced value, then (from the cache) for the split; 8 rows' 16-byte stores are 128 contiguous bytes.
__global__ void __launch_bounds__(256) split_a_kernel(int64_t M, int K, int nslab, const float2* __restrict__ A,
                                                      int64_t lda, const int* __restrict__ dk,
                                                      unsigned char* __restrict__ out, float* __restrict__ inv,
                                                      int64_t rows_pad) {
  const int lane = threadIdx.x & 31;
  const int64_t row = (int64_t(blockIdx.x) * 8 + (threadIdx.x >> 5)) * 8 + (lane & 7);
  if (row >= rows_pad) return;  // (rows_pad is a multiple of 128: whole warps)
  const float2* a = A + row * lda;
  const bool ok = row < M;
  const int dmax = balance_max(dk, lane);
  int e = kNone;
  for (int g = lane >> 3; g < 2 * nslab; g += 4) {
    int d[8];
    balance8(dk, 8 * g, dmax, d);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = 8 * g + i;
      const float2 v = ok && k < K ? a[k] : make_float2(0.f, 0.f);
      e = max(e, value_exp(v) + d[i]);
    }
  }
  e = max(e, __shfl_xor_sync(0xffffffffu, e, 8));
  e = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
  const int sh = scale_exp(e);
  if (lane < 8) inv[row] = pow2(-sh);
  unsigned char* base = out + (row / U_TM) * nslab * int64_t(U_ABYTES);
  for (int g = lane >> 3; g < 2 * nslab; g += 4) {
    float re[8], im[8];
    int d[8];
    balance8(dk, 8 * g, dmax, d);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = 8 * g + i;
      const float2 v = ok && k < K ? a[k] : make_float2(0.f, 0.f);
      re[i] = scale2(v.x, sh + d[i]);
      im[i] = scale2(v.y, sh + d[i]);
    }
    uint4 rh, rl, ih, il;
    split8(re, rh, rl);
    split8(im, ih, il);
    unsigned char* o = base + (g >> 1) * int64_t(U_ABYTES) + part_off(int(row % U_TM), (g & 1) * 8);
    *reinterpret_cast<uint4*>(o) = rh;
    *reinterpret_cast<uint4*>(o + U_PART) = rl;
    *reinterpret_cast<uint4*>(o + 2 * U_PART) = ih;
    *reinterpret_cast<uint4*>(o + 3 * U_PART) = il;
  }
}
// B (K x N, ldb), K <= 256: out[(ct * nslab + s) * 24 KB + p * 4 KB + part_off(c, k)], parts
// Br_h, Bi_h, -Br_h, Br_l, Bi_l, -Br_l; zero outside K x N; inv[col] the inverse scales.  A CTA per
// 32 columns, lanes along the columns (coalesced), the warps sharing the groups of 8 values of k, first for the
// columns' largest balanced values, then for the split.
__global__ void __launch_bounds__(256) split_b_kernel(int64_t N, int K, int nslab, const float2* __restrict__ B,
                                                      int64_t ldb, const int* __restrict__ dk,
                                                      unsigned char* __restrict__ out, float* __restrict__ inv) {
  __shared__ int s_e[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t col = int64_t(blockIdx.x) * 32 + lane;
  const bool ok = col < N;
  const int dmax = balance_max(dk, lane);
  int e = kNone;
  for (int g = warp; g < 2 * nslab; g += 8) {
    int d[8];
    balance8(dk, 8 * g, dmax, d);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = 8 * g + i;
      const float2 v = ok && k < K ? B[int64_t(k) * ldb + col] : make_float2(0.f, 0.f);
      e = max(e, value_exp(v) - d[i]);
    }
  }
  s_e[warp][lane] = e;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) e = max(e, s_e[w][lane]);
  const int sh = scale_exp(e);
  if (warp == 0) inv[col] = pow2(-sh);
  unsigned char* base = out + (col / U_TN) * nslab * int64_t(U_BBYTES);
  for (int g = warp; g < 2 * nslab; g += 8) {
    float re[8], im[8];
    int d[8];
    balance8(dk, 8 * g, dmax, d);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = 8 * g + i;
      const float2 v = ok && k < K ? B[int64_t(k) * ldb + col] : make_float2(0.f, 0.f);
      re[i] = scale2(v.x, sh - d[i]);
      im[i] = scale2(v.y, sh - d[i]);
    }
    uint4 rh, rl, ih, il;
    split8(re, rh, rl);
    split8(im, ih, il);
    unsigned char* o = base + (g >> 1) * int64_t(U_BBYTES) + part_off(int(col % U_TN), (g & 1) * 8);
    *reinterpret_cast<uint4*>(o) = rh;
    *reinterpret_cast<uint4*>(o + U_PART) = ih;
    *reinterpret_cast<uint4*>(o + 2 * U_PART) = neg8(rh);
    *reinterpret_cast<uint4*>(o + 3 * U_PART) = rl;
    *reinterpret_cast<uint4*>(o + 4 * U_PART) = il;
    *reinterpret_cast<uint4*>(o + 5 * U_PART) = neg8(rl);
  }
}

// tile index -> (row tile, column tile): super-rows of U_GROUP row tiles, columns inside
__device__ __forceinline__ void tile_rc(int64_t tile, int64_t RT, int64_t CT, int64_t& rt, int64_t& ct) {
  const int64_t g = tile / (int64_t(U_GROUP) * CT);
  const int64_t local = tile - g * U_GROUP * CT;
  const int64_t gr = min(int64_t(U_GROUP), RT - g * U_GROUP);
  ct = local / gr;
  rt = g * U_GROUP + local % gr;
}

// ---------------------------------------------------------------- the update
__global__ void __launch_bounds__(U_THREADS, 1)
    cgemm_update_split_kernel(int64_t M, int64_t N, int nslab, const unsigned char* __restrict__ As,
                              const unsigned char* __restrict__ Bs, const float* __restrict__ inv_a,
                              const float* __restrict__ inv_b, float2* __restrict__ C, int64_t ldc, int* status,
                              int vec_ok) {
  extern __shared__ unsigned char u_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(u_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t bar_full[U_STAGES], bar_empty[U_STAGES], bar_tfull[2], bar_tempty[2], bar_drain;
  __shared__ uint32_t tmem_sh;
  __shared__ volatile int abort_sh;
  __shared__ volatile int epi_stop[2];
  __shared__ float s_inv_b[2][U_TN];  // the column scales of each epilogue group's tile
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t RT = (M + U_TM - 1) / U_TM, CT = (N + U_TN - 1) / U_TN, tiles = RT * CT;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_sh)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < U_STAGES; ++i) {
      u_init(su32(&bar_full[i]), 1);
      u_init(su32(&bar_empty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      u_init(su32(&bar_tfull[i]), 1);
      u_init(su32(&bar_tempty[i]), 256);
    }
    u_init(su32(&bar_drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
    abort_sh = 0;
    epi_stop[0] = epi_stop[1] = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_sh;
  auto fail = [&]() {
    abort_sh = 1;
    atomicExch(status, FOSB_ERR_TIMEOUT);
  };

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int64_t it = 0;
      for (int64_t tile = blockIdx.x; tile < tiles && !abort_sh; tile += gridDim.x) {
        int64_t rt, ct;
        tile_rc(tile, RT, CT, rt, ct);
        for (int s = 0; s < nslab; ++s, ++it) {
          const int st = int(it % U_STAGES);
          const int64_t use = it / U_STAGES;
          if (use > 0 && !u_wait(su32(&bar_empty[st]), uint32_t((use - 1) & 1))) {
            fail();
            break;
          }
          unsigned char* sa = smem + st * U_STAGE;
          const uint32_t fb = su32(&bar_full[st]);
          u_expect_tx(fb, U_STAGE);
          u_bulk(su32(sa), As + (rt * nslab + s) * int64_t(U_ABYTES), U_ABYTES, fb);
          u_bulk(su32(sa + U_ABYTES), Bs + (ct * nslab + s) * int64_t(U_BBYTES), U_BBYTES, fb);
        }
      }
      // wait for every copy issued here that the MMA thread may not have consumed
      for (int64_t j = it > U_STAGES ? it - U_STAGES : 0; j < it; ++j)
        if (!u_wait(su32(&bar_full[int(j % U_STAGES)]), uint32_t((j / U_STAGES) & 1))) fail();
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      const uint32_t id = u_idesc(false), idn = u_idesc(true);
      int64_t it = 0, tcount = 0;
      for (int64_t tile = blockIdx.x; tile < tiles && !abort_sh; tile += gridDim.x, ++tcount) {
        const int b = int(tcount & 1);
        const int64_t ub = tcount >> 1;
        if (ub > 0 && !u_wait(su32(&bar_tempty[b]), uint32_t((ub - 1) & 1))) {
          fail();
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t d = tmem + uint32_t(b) * 256;
        for (int s = 0; s < nslab; ++s, ++it) {
          const int st = int(it % U_STAGES);
          const int64_t use = it / U_STAGES;
          if (!u_wait(su32(&bar_full[st]), uint32_t(use & 1))) {
            fail();
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t a0 = su32(smem + st * U_STAGE), b0 = a0 + U_ABYTES;
          const uint64_t arb = sdesc(a0), ars = sdesc(a0 + U_PART), aib = sdesc(a0 + 2 * U_PART),
                         ais = sdesc(a0 + 3 * U_PART);
          // B windows: [Br | Bi] at part 0 (big) / 3 (small); [Bi | -Br] at part 1 / 4
          const uint64_t w1b = sdesc(b0), w1s = sdesc(b0 + 3 * U_PART);
          const uint64_t w2b = sdesc(b0 + U_PART), w2s = sdesc(b0 + 4 * U_PART);
          const uint32_t acc0 = s > 0 ? 1u : 0u;
          u_mma(d, arb, w1b, id, acc0);
          u_mma(d, arb, w1s, id, 1u);
          u_mma(d, ars, w1b, id, 1u);
          u_mma(d, aib, w2b, idn, 1u);
          u_mma(d, aib, w2s, idn, 1u);
          u_mma(d, ais, w2b, idn, 1u);
          u_commit(su32(&bar_empty[st]));
        }
        if (abort_sh) break;
        u_commit(su32(&bar_tfull[b]));
      }
      u_commit(su32(&bar_drain));  // completes once every MMA issued above has finished
      if (!u_wait(su32(&bar_drain), 0u)) fail();
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue (warps 2-9)
    // Two groups of four warps, each with its own buffer and barrier, take the 32-column quarters
    // g and g + 2 of a tile: the quarter of C is copied into the padded shared tile by cp.async (for
    // the first quarter issued before the accumulator wait), thread r subtracts its TMEM row (lane
    // r) in place, and the quarter is stored with coalesced 16-byte writes.  One group on 64-column
    // halves left the tensor pipe 44 % active: a half's way from and to memory took longer than its
    // MMAs.  Without 16-byte alignment of C the tile takes the negated accumulator and C is updated
    // element by element.
    const int grp = (warp - 2) >> 2;
    const int et = tid - 2 * 32 - grp * 128;  // 0..127
    const int lane_base = (warp & 3) * 32;    // TMEM lane quarter of this warp
    const int r_local = lane_base + lane;
    float2* sE = reinterpret_cast<float2*>(smem + U_EPI_OFF) + grp * (U_TM * U_EPI_LD);
    float* s_scale = s_inv_b[grp];
    int64_t tcount = 0;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++tcount) {
      const int b = int(tcount & 1);
      const int64_t ub = tcount >> 1;
      int64_t rt, ct;
      tile_rc(tile, RT, CT, rt, ct);
      const int64_t row0 = rt * U_TM, col0 = ct * U_TN;
      const uint32_t d = tmem + uint32_t(b) * 256 + (uint32_t(lane_base) << 16);
      const float sa = -inv_a[row0 + r_local];
      s_scale[et] = inv_b[col0 + et];  // read after the barrier below; the last tile's reads are behind one
#pragma unroll 1
      for (int h = grp; h < 4; h += 2) {
        const int64_t gc0 = col0 + h * U_EPI_N;
        if (vec_ok) {
#pragma unroll 8
          for (int q = 0; q < U_EPI_N / 2; ++q) {
            const int e = et + 128 * q;  // 0 .. 2047 pairs of complex
            const int r = e / (U_EPI_N / 2), c = (e % (U_EPI_N / 2)) * 2;
            const int64_t gr = row0 + r, gc = gc0 + c;
            const int bytes = gr < M ? (gc + 1 < N ? 16 : (gc < N ? 8 : 0)) : 0;
            u_cp16(su32(&sE[u_piece(r, c >> 1)]), bytes ? static_cast<const void*>(C + gr * ldc + gc) : C, bytes);
          }
          u_cp_commit();
        }
        if (h == grp) {
          // the stop decision must be the same in all four warps (they share named barriers)
          if (!u_wait(su32(&bar_tfull[b]), uint32_t(ub & 1))) {
            fail();
            epi_stop[grp] = 1;
          }
          u_bar(1 + grp, 128);
          if (epi_stop[grp]) {
            u_cp_wait_all();  // no copy may land after the kernel has left
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
        }
        if (vec_ok) {
          u_cp_wait_all();
          u_bar(1 + grp, 128);  // every thread's pieces of C are in the tile
        }
        {
          uint32_t vr[32], vi[32];
          u_ld32(d + h * U_EPI_N, vr);
          u_ld32(d + 128 + h * U_EPI_N, vi);
          asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
          for (int j = 0; j < U_EPI_N; j += 2) {
            float4* p = reinterpret_cast<float4*>(&sE[u_piece(r_local, j >> 1)]);
            float4 c4 = vec_ok ? *p : make_float4(0.f, 0.f, 0.f, 0.f);
            // (acc 2^-ea) 2^-eb: two exact scalings, so neither product of scales can overflow
            const float s0 = s_scale[h * U_EPI_N + j], s1 = s_scale[h * U_EPI_N + j + 1];
            c4.x = fmaf(__uint_as_float(vr[j]) * sa, s0, c4.x);
            c4.y = fmaf(__uint_as_float(vi[j]) * sa, s0, c4.y);
            c4.z = fmaf(__uint_as_float(vr[j + 1]) * sa, s1, c4.z);
            c4.w = fmaf(__uint_as_float(vi[j + 1]) * sa, s1, c4.w);
            *p = c4;
          }
        }
        if (h >= 2) {  // every accumulator value of this group's quarters has been read
          asm volatile("tcgen05.fence::before_thread_sync;");
          u_arrive(su32(&bar_tempty[b]));
        }
        u_bar(1 + grp, 128);
        if (vec_ok) {
#pragma unroll 8
          for (int q = 0; q < U_EPI_N / 2; ++q) {
            const int e = et + 128 * q;
            const int r = e / (U_EPI_N / 2), c = (e % (U_EPI_N / 2)) * 2;
            const int64_t gr = row0 + r, gc = gc0 + c;
            if (gr < M && gc + 1 < N) {
              *reinterpret_cast<float4*>(C + gr * ldc + gc) = *reinterpret_cast<const float4*>(&sE[u_piece(r, c >> 1)]);
            } else if (gr < M && gc < N) {
              C[gr * ldc + gc] = sE[u_piece(r, c >> 1)];
            }
          }
        } else {
#pragma unroll 4
          for (int q = 0; q < U_EPI_N; ++q) {
            const int e = et + 128 * q;  // 0 .. 4095
            const int r = e / U_EPI_N, c = e % U_EPI_N;
            const int64_t gr = row0 + r, gc = gc0 + c;
            if (gr < M && gc < N) {  // the tile holds -D here: C += it
              const float2 dd = sE[u_piece(r, c >> 1) + (c & 1)];
              float2 o = C[gr * ldc + gc];
              o.x += dd.x;
              o.y += dd.y;
              C[gr * ldc + gc] = o;
            }
          }
        }
        u_bar(1 + grp, 128);  // the buffer is free for the next quarter's copies
      }
      if (epi_stop[grp]) break;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

inline unsigned ucdiv(int64_t a, int64_t b) { return unsigned((a + b - 1) / b); }

}  // namespace

// the image, then one scale per padded row or column; behind B's also the balance exponents
size_t update_split_a_bytes(int64_t M) {
  return size_t((M + U_TM - 1) / U_TM) * (size_t(U_SLABS) * U_ABYTES + U_TM * sizeof(float));
}
size_t update_split_b_bytes(int64_t N) {
  return size_t((N + U_TN - 1) / U_TN) * (size_t(U_SLABS) * U_BBYTES + U_TN * sizeof(float)) + U_KB * sizeof(int);
}

// C (M x N) -= A (M x K) B (K x N), complex64 row-major, K <= kLuBlock: split A and B once into
// the workspaces (update_split_a_bytes(M), update_split_b_bytes(N) bytes, 16-byte aligned),
// then the bulk-copy-fed tcgen05 update.  col_ex: the biased FP32 exponents of the scale of C's columns.
cudaError_t cgemm_update_tc_split(int64_t M, int64_t N, int64_t K, const void* A, int64_t lda, const void* B,
                                  int64_t ldb, void* C, int64_t ldc, int* status, void* ws_a, void* ws_b,
                                  const int* col_ex, cudaStream_t s) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  if (K > U_KB) return cudaErrorInvalidValue;
  static bool attr[64] = {};
  static int nsm[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr[dev]) {
    cudaError_t e = cudaFuncSetAttribute(cgemm_update_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, U_SMEM);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&nsm[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    attr[dev] = true;
  }
  const int64_t RT = (M + U_TM - 1) / U_TM, CT = (N + U_TN - 1) / U_TN;
  const int64_t rows_pad = RT * U_TM, cols_pad = CT * U_TN;
  ProfScope prof("lu_update", s, 8.0 * double(M) * double(N) * double(K));  // the splits are part of it
  const int nslab = int((K + U_KS - 1) / U_KS);  // tiles packed with exactly nslab slabs each
  unsigned char* img_a = static_cast<unsigned char*>(ws_a);
  unsigned char* img_b = static_cast<unsigned char*>(ws_b);
  float* inv_a = reinterpret_cast<float*>(img_a + RT * nslab * int64_t(U_ABYTES));
  float* inv_b = reinterpret_cast<float*>(img_b + CT * nslab * int64_t(U_BBYTES));
  int* dk = reinterpret_cast<int*>(inv_b + cols_pad);
  const float2 *a = static_cast<const float2*>(A), *b = static_cast<const float2*>(B);
  row_balance_kernel<<<U_KB, 512, 0, s>>>(N, int(K), b, ldb, col_ex, dk);
  split_a_kernel<<<ucdiv(rows_pad, 64), 256, 0, s>>>(M, int(K), nslab, a, lda, dk, img_a, inv_a, rows_pad);
  split_b_kernel<<<ucdiv(cols_pad, 32), 256, 0, s>>>(N, int(K), nslab, b, ldb, dk, img_b, inv_b);
  note_launches(3);
  const unsigned grid = unsigned(std::min<int64_t>(RT * CT, std::max(nsm[dev], 1)));
  const int vec_ok = (reinterpret_cast<uintptr_t>(C) % 16 == 0) && (ldc % 2 == 0);
  cgemm_update_split_kernel<<<grid, U_THREADS, U_SMEM, s>>>(M, N, nslab, img_a, img_b, inv_a, inv_b,
                                                          static_cast<float2*>(C), ldc, status, vec_ok);
  return launched();
}

}  // namespace fosb
