// Streaming triangular solves with complex64 factors (A6: the forward and backward sweeps
// L y = P b, U x = y of every refined solve, and of the multi-right-hand-side covariance solves).
//
// A blocked sweep that launches one diagonal solve and one panel update per 64-row block
// is latency-bound (2 x n/64 dependent launches per sweep).  Here one persistent kernel
// does a whole sweep.  The right-hand sides are cut into chunks of 1, 2, 4 or 8 columns
// (chunk_width; the last chunk may have fewer); CTAs take (block, chunk) tasks in block-major order
// from a ticket counter.  With D_i the inverse of the diagonal block and j the blocks that
// precede i in the sweep, the last of them h,
//     y_i = D_i (x_i - sum_{j != h} L_ij y_j) - E_i y_h,   E_i = D_i L_ih  (E_i formed once per factorisation),
// so between y_h and y_i there is one 64 x 64 product and not two; everything else of a task
// is done while y_h is still on its way.  The solution carries its own readiness: the output
// is filled with a bit pattern that no arithmetic result has (both words all ones, a NaN
// that the hardware never returns) and a waiting thread polls the very values it needs with
// 8-byte loads, so a block costs one store and one load of latency instead of a fence, a flag
// and a second read.
//
// With many right-hand sides the tile products bound the sweep, not the chain: then the kernel
// solves 512 rows at a time and the rows behind them are updated on the tensor cores
// (cgemm_update_tc, K = 512) before the next 512.
//  A task only waits for tasks that were taken earlier, by CTAs that are
// running or done, so the waits always end; each is bounded anyway and a time-out sets the
// status word, which every waiter polls, so the sweep ends quickly and the host reports
// FOSB_ERR_TIMEOUT.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "fosb_internal.h"

namespace fosb {
namespace {

constexpr int kTB = 64;                         // rows per block
constexpr long long kFlagSpinLimit = 1ll << 26;
// Poll limit of the waits on this device (kFlagSpinLimit unless changed by
// fosb_debug_set_wait_limit).
__device__ long long g_flag_wait_limit = kFlagSpinLimit;

__device__ __forceinline__ void cfma(float2& acc, float2 a, float2 b) {  // acc += a b
  acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
  acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
}

// Inverse of each 64 x 64 diagonal block of the factors (unit lower L_ii for which = 0,
// upper U_ii for which = 1), row-major in Dinv[i][64][64]: one CTA per block, each warp
// substitutes 8 unit columns.  Used by the streaming sweeps so that the critical path of a
// block is a parallel 64 x 64 matrix-vector product instead of a 64-step substitution.
__global__ void __launch_bounds__(256) tri_block_inverse_kernel(const float2* __restrict__ LU, int64_t n, int64_t ld,
                                                                int which, float2* __restrict__ Dinv) {
  __shared__ float2 sDt[kTB][kTB + 1];  // sDt[k][r] = D[r][k]
  const int64_t ib = blockIdx.x, r0 = ib * kTB;
  const int rows = int(std::min<int64_t>(kTB, n - r0));
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int e = t; e < kTB * kTB; e += blockDim.x) {
    const int rr = e / kTB, kk = e % kTB;
    sDt[kk][rr] = (rr < rows && kk < rows) ? LU[(r0 + rr) * ld + r0 + kk] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  float2* out = Dinv + ib * kTB * kTB;
  const float2 zero = make_float2(0.f, 0.f);
  for (int cidx = 0; cidx < 8; ++cidx) {
    const int col = warp * 8 + cidx;  // column of the inverse: solve D x = e_col
    float2 x0 = lane == col ? make_float2(1.f, 0.f) : zero;
    float2 x1 = lane + 32 == col ? make_float2(1.f, 0.f) : zero;
    if (col >= rows) {
      x0 = x1 = zero;
    } else if (which == 0) {
      for (int i = 0; i < rows - 1; ++i) {
        float2 xi = i < 32 ? x0 : x1;
        xi.x = __shfl_sync(0xffffffffu, xi.x, i & 31);
        xi.y = __shfl_sync(0xffffffffu, xi.y, i & 31);
        if (lane > i && lane < rows) {
          const float2 d = sDt[i][lane];
          x0.x -= d.x * xi.x - d.y * xi.y;
          x0.y -= d.x * xi.y + d.y * xi.x;
        }
        if (lane + 32 > i && lane + 32 < rows) {
          const float2 d = sDt[i][lane + 32];
          x1.x -= d.x * xi.x - d.y * xi.y;
          x1.y -= d.x * xi.y + d.y * xi.x;
        }
      }
    } else {
      for (int i = rows - 1; i >= 0; --i) {
        const float2 d = sDt[i][i];
        const float den = d.x * d.x + d.y * d.y;
        const bool mine0 = i < 32 && lane == i, mine1 = i >= 32 && lane == i - 32;
        if (mine0 || mine1) {
          const float2 v = mine0 ? x0 : x1;
          const float2 qv =
              den > 0.f ? make_float2((v.x * d.x + v.y * d.y) / den, (v.y * d.x - v.x * d.y) / den) : zero;
          if (mine0) x0 = qv; else x1 = qv;
        }
        float2 xi = i < 32 ? x0 : x1;
        xi.x = __shfl_sync(0xffffffffu, xi.x, i & 31);
        xi.y = __shfl_sync(0xffffffffu, xi.y, i & 31);
        if (lane < i) {
          const float2 dd = sDt[i][lane];
          x0.x -= dd.x * xi.x - dd.y * xi.y;
          x0.y -= dd.x * xi.y + dd.y * xi.x;
        }
        if (lane + 32 < i) {
          const float2 dd = sDt[i][lane + 32];
          x1.x -= dd.x * xi.x - dd.y * xi.y;
          x1.y -= dd.x * xi.y + dd.y * xi.x;
        }
      }
    }
    out[lane * kTB + col] = x0;  // Dinv[row][col]
    out[(lane + 32) * kTB + col] = x1;
  }
}

// E_i = D_i L_ih (which = 0: h = i - 1; which = 1, U: h = i + 1), one CTA per block; zero where
// there is no such neighbour.
__global__ void __launch_bounds__(256) tri_neighbour_kernel(const float2* __restrict__ LU, int64_t n, int64_t ld,
                                                            int which, const float2* __restrict__ Dinv,
                                                            float2* __restrict__ E) {
  extern __shared__ float4 nb_raw[];
  auto sD = reinterpret_cast<float2 (*)[kTB + 1]>(nb_raw);  // D, then the tile
  auto sT = sD + kTB;
  const int64_t ib = blockIdx.x, nblk = (n + kTB - 1) / kTB, hb = which ? ib + 1 : ib - 1;
  const int64_t r0 = ib * kTB, c0 = hb * kTB;
  const bool any = hb >= 0 && hb < nblk;
  for (int e = threadIdx.x; e < kTB * kTB; e += blockDim.x) {
    const int r = e / kTB, c = e % kTB;
    sD[r][c] = Dinv[ib * kTB * kTB + e];
    sT[r][c] = any && r0 + r < n && c0 + c < n ? LU[(r0 + r) * ld + c0 + c] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  const int r = threadIdx.x >> 2, cq = threadIdx.x & 3;  // row r, columns cq, cq + 4, ...
  float2 acc[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) acc[c] = make_float2(0.f, 0.f);
  for (int k = 0; k < kTB; ++k) {
    const float2 d = sD[r][k];
#pragma unroll
    for (int c = 0; c < 16; ++c) cfma(acc[c], d, sT[k][cq + 4 * c]);
  }
#pragma unroll
  for (int c = 0; c < 16; ++c) E[(ib * kTB + r) * kTB + cq + 4 * c] = acc[c];
}

// One step of refinement of the inverses, D += D (I - A D) with A the diagonal block and the residual in
// float-float, for solves that nothing refines afterwards (complex64 factorisations).  D then
// carries one rounding instead of the errors of 64 substitution steps.  Such sweeps also do without E,
// whose products cancel against D x: complex64 solves, random matrices, largest componentwise
// backward error at n = 120 / 480: 3.5e-6 / 4.7e-6 with E, 1.5e-6 / 2.6e-6 with E and D refined, 7.8e-7 /
// 1.7e-6 with D refined and no E (1.4e-6 / 2.3e-6 with an unrefined D and no E).
__global__ void __launch_bounds__(256) tri_refine_kernel(const float2* __restrict__ LU, int64_t n, int64_t ld, int which,
                                                         float2* Dinv) {
  extern __shared__ float4 nb_raw[];
  auto sA = reinterpret_cast<float2 (*)[kTB + 1]>(nb_raw);
  auto sD = sA + kTB, sR = sD + kTB;
  const int64_t ib = blockIdx.x, r0 = ib * kTB;
  const int rows = int(std::min<int64_t>(kTB, n - r0));
  for (int e = threadIdx.x; e < kTB * kTB; e += blockDim.x) {
    const int r = e / kTB, c = e % kTB;
    float2 a = make_float2(0.f, 0.f);
    if (r < rows && c < rows && (which ? c >= r : c < r)) a = LU[(r0 + r) * ld + r0 + c];
    if (!which && r == c) a = make_float2(1.f, 0.f);
    sA[r][c] = a;
    sD[r][c] = Dinv[ib * kTB * kTB + e];
  }
  __syncthreads();
  const int r = threadIdx.x >> 2, cq = threadIdx.x & 3, warp = threadIdx.x >> 5;  // columns cq, cq + 4, ...
  const int k0 = which ? 8 * warp : 0, k1 = which ? kTB : 8 * warp + 8;              // A and D are triangular
  float2 re[16], im[16];                                                            // (hi, lo)
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    re[c] = make_float2(r == cq + 4 * c && r < rows ? 1.f : 0.f, 0.f);
    im[c] = make_float2(0.f, 0.f);
  }
  auto sub = [](float2& s, float p, float q) {  // s -= p q
    const float v = -p * q, e = fmaf(-p, q, -v), t = s.x + v, b = t - s.x;
    s.y += ((s.x - (t - b)) + (v - b)) + e;
    s.x = t;
  };
  for (int k = k0; k < k1; ++k) {
    const float2 a = sA[r][k];
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const float2 x = sD[k][cq + 4 * c];
      sub(re[c], a.x, x.x);
      sub(re[c], -a.y, x.y);
      sub(im[c], a.x, x.y);
      sub(im[c], a.y, x.x);
    }
  }
#pragma unroll
  for (int c = 0; c < 16; ++c) sR[r][cq + 4 * c] = make_float2(re[c].x + re[c].y, im[c].x + im[c].y);
  __syncthreads();
  float2 acc[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) acc[c] = make_float2(0.f, 0.f);
  for (int k = k0; k < k1; ++k) {
    const float2 d = sD[r][k];
#pragma unroll
    for (int c = 0; c < 16; ++c) cfma(acc[c], d, sR[k][cq + 4 * c]);
  }
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    const float2 x = sD[r][cq + 4 * c];
    Dinv[(ib * kTB + r) * kTB + cq + 4 * c] = make_float2(x.x + acc[c].x, x.y + acc[c].y);
  }
}

// Shared tiles of the streaming sweep.  A factor tile (later the inverse of the diagonal block)
// and the neighbour product E are 64 x 64 with a row pitch of 72 complex values; the published
// blocks of the solution are 64 x NR with a pitch that keeps 16-byte rows of 4 and 8 columns in
// distinct banks.  Thread (g, q) of 256 owns rows g and g + 32 and the columns q, q + 8,
// ..., q + 56, so in one step of c the 16 threads of a half-warp read 8 consecutive complex
// values of two rows 72 apart (every bank once) and 8 rows of the solution block (distinct banks).
constexpr int kLP = 72;
template <int NR>
struct StreamSmem {
  static constexpr int NRP = NR <= 2 ? NR : NR + 2;
  float2 L[kTB][kLP];
  float2 E[kTB][kLP];
  float2 Y[2][kTB][NRP];  // the current block of the solution; minus the neighbour's
};

// acc0/acc1 (rows g, g + 32) += T[rows][cols] Y[cols][0..NR) over this thread's 8 columns
template <int NR>
__device__ __forceinline__ void stream_tile_product(const float2 (*T)[kLP], const float2 (*Y)[StreamSmem<NR>::NRP],
                                                    int g, int q, float2 (&acc0)[NR], float2 (&acc1)[NR]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int cc = q + 8 * c;
    const float2 l0 = T[g][cc], l1 = T[g + 32][cc];
    if constexpr (NR % 2 == 0) {
#pragma unroll
      for (int k = 0; k < NR; k += 2) {
        const float4 y = *reinterpret_cast<const float4*>(&Y[cc][k]);
        const float2 ya = make_float2(y.x, y.y), yb = make_float2(y.z, y.w);
        cfma(acc0[k], l0, ya);
        cfma(acc1[k], l1, ya);
        cfma(acc0[k + 1], l0, yb);
        cfma(acc1[k + 1], l1, yb);
      }
    } else {
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        const float2 y = Y[cc][k];
        cfma(acc0[k], l0, y);
        cfma(acc1[k], l1, y);
      }
    }
  }
}
// Sum over the 8 column owners q (lanes differing in their low three bits), scattered: lane q is
// left with row g + 32 (q & 1) and the right-hand sides from (q >> 1) NR/4 on (NR % 4 == 0; each
// halving step sends one half and keeps the other), or with both rows in lane q = 0.
template <int NR>
struct StreamOut {
  static constexpr bool kSplit = NR % 4 == 0;
};
template <int NR>
__device__ __forceinline__ void stream_reduce(float2 (&a0)[NR], float2 (&a1)[NR], int q) {
  auto add = [](float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); };
  auto swap2 = [](float2 v, int off) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, off), __shfl_xor_sync(0xffffffffu, v.y, off));
  };
  if constexpr (StreamOut<NR>::kSplit) {
#pragma unroll
    for (int k = 0; k < NR; ++k) {  // rows
      const float2 keep = q & 1 ? a1[k] : a0[k], give = q & 1 ? a0[k] : a1[k];
      a0[k] = add(keep, swap2(give, 1));
    }
#pragma unroll
    for (int k = 0; k < NR / 2; ++k) {  // halves of the right-hand sides
      const float2 keep = q & 4 ? a0[k + NR / 2] : a0[k], give = q & 4 ? a0[k] : a0[k + NR / 2];
      a0[k] = add(keep, swap2(give, 4));
    }
#pragma unroll
    for (int k = 0; k < NR / 4; ++k) {  // quarters
      const float2 keep = q & 2 ? a0[k + NR / 4] : a0[k], give = q & 2 ? a0[k] : a0[k + NR / 4];
      a0[k] = add(keep, swap2(give, 2));
    }
  } else {
#pragma unroll
    for (int k = 0; k < NR; ++k)
#pragma unroll
      for (int off = 1; off < 8; off <<= 1) {
        a0[k] = add(a0[k], swap2(a0[k], off));
        a1[k] = add(a1[k], swap2(a1[k], off));
      }
  }
}
// visits the (row, right-hand side, value) that this lane is left with
template <int NR, class Fn>
__device__ __forceinline__ void stream_each(const float2 (&a0)[NR], const float2 (&a1)[NR], int g, int q, Fn fn) {
  if constexpr (StreamOut<NR>::kSplit) {
#pragma unroll
    for (int k = 0; k < NR / 4; ++k) fn(g + 32 * (q & 1), (q >> 1) * (NR / 4) + k, a0[k]);
  } else if (q == 0) {
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      fn(g, k, a0[k]);
      fn(g + 32, k, a1[k]);
    }
  }
}

constexpr unsigned long long kNotReady = ~0ull;
__device__ __forceinline__ unsigned long long ld_relaxed(const float2* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(float2* p, float2 v) {
  const unsigned long long b = (static_cast<unsigned long long>(__float_as_uint(v.y)) << 32) | __float_as_uint(v.x);
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(b) : "memory");
}

// Blocks first .. first + count - 1 of the sweep (in its order) on their own: x are the right-hand
// sides (n x nrhs, rows ldx apart) less everything that earlier blocks contribute, y the solution, all ones
// (kNotReady) on entry.
// Chain-bound: a block's latency is one store-to-load trip, a product and a reduction.
// One sweep at N = 15360: 0.36 ms for 1 column, 0.82 for 16 (1.32 and 3.01 with a flag per block, the
// diagonal solve behind the last product and chunks of 16 columns).
template <int NR>
__global__ void __launch_bounds__(256, 2)
    trsv_stream_kernel(const float2* __restrict__ LU, int64_t n, int64_t ld, const float2* __restrict__ Dinv,
                       const float2* __restrict__ E, const float2* __restrict__ x, float2* y, int64_t nrhs, int64_t ldx, int64_t chunks,
                       int64_t first, int64_t count, int upper, int use_e, int* ticket, int* status) {
  extern __shared__ float4 stream_raw[];
  StreamSmem<NR>& sm = *reinterpret_cast<StreamSmem<NR>*>(stream_raw);
  __shared__ long long s_task;
  __shared__ int s_abort;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int g = t >> 3, q = t & 7;
  const int64_t nblk = (n + kTB - 1) / kTB;
  constexpr int kPer = (kTB * NR + 255) / 256;  // values of a solution block per thread
  const long long limit = g_flag_wait_limit;
  for (;;) {
    __syncthreads();  // every thread is done with the last task
    if (t == 0) {
      s_task = atomicAdd(ticket, 1);
      s_abort = 0;
    }
    __syncthreads();
    const int64_t task = s_task;
    const int64_t b = task / chunks;
    if (b >= count) break;
    auto block_at = [&](int64_t p) { return upper ? nblk - 1 - first - p : first + p; };
    const int64_t ib = block_at(b);
    const int64_t r0 = ib * kTB;
    const int rows = int(std::min<int64_t>(kTB, n - r0));
    const int64_t k0 = (task % chunks) * NR;
    const int nc = int(std::min<int64_t>(NR, nrhs - k0));  // this chunk's columns
    const int64_t far = use_e && b > 0 ? b - 1 : b;        // blocks that come in through their tiles
    if (far < b) {
      const float2* e = E + ib * kTB * kTB;
#pragma unroll
      for (int i = 0; i < kTB * kTB / 512; ++i) {
        const int p = t + 256 * i, r = p >> 5, c = (p & 31) * 2;  // 16-byte pieces
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         static_cast<uint32_t>(__cvta_generic_to_shared(&sm.E[r][c]))),
                     "l"(e + r * kTB + c)
                     : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    float2 acc0[NR], acc1[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) acc0[k] = acc1[k] = make_float2(0.f, 0.f);
    // factor tile jj (the far blocks in publication order, then the inverse of the diagonal block)
    // in registers: warp w holds rows 8w .. 8w+7, lanes the columns lane and lane + 32
    float2 lreg[16];
    auto fetch = [&](int64_t jj) {
      const bool diag = jj >= far;
      const int64_t c0 = diag ? 0 : block_at(jj) * kTB;
      const float2* base = diag ? Dinv + ib * kTB * kTB : LU + r0 * ld + c0;
      const int64_t pitch = diag ? kTB : ld;
      const int rr_n = diag ? kTB : rows, cols = diag ? kTB : int(std::min<int64_t>(kTB, n - c0));
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int rr = warp * 8 + i;
        const float2* src = base + rr * pitch;
        lreg[2 * i] = (rr < rr_n && lane < cols) ? __ldg(src + lane) : make_float2(0.f, 0.f);
        lreg[2 * i + 1] = (rr < rr_n && lane + 32 < cols) ? __ldg(src + lane + 32) : make_float2(0.f, 0.f);
      }
    };
    auto store_tile = [&]() {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        sm.L[warp * 8 + i][lane] = lreg[2 * i];
        sm.L[warp * 8 + i][lane + 32] = lreg[2 * i + 1];
      }
    };
    // waits for this thread's values of solution block jj (publication order)
    float2 v[kPer];
    auto poll = [&](int64_t jj) {
      const int64_t c0 = block_at(jj) * kTB;
      const int cols = int(std::min<int64_t>(kTB, n - c0));
      long long spins = 0;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int e = t + 256 * i, rr = e / NR, k = e % NR;
        v[i] = make_float2(0.f, 0.f);
        if (rr >= cols || k >= nc) continue;
        const float2* p = y + (c0 + rr) * ldx + k0 + k;
        unsigned long long w = ld_relaxed(p);
        while (w == kNotReady) {
          if (++spins > limit || *(volatile int*)status == FOSB_ERR_TIMEOUT) {
            atomicExch(status, FOSB_ERR_TIMEOUT);
            s_abort = 1;
            return;
          }
          w = ld_relaxed(p);
        }
        v[i] = make_float2(__uint_as_float(unsigned(w)), __uint_as_float(unsigned(w >> 32)));
      }
    };
    auto store_y = [&](float2 (*Y)[StreamSmem<NR>::NRP], float sign) {
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int e = t + 256 * i;
        if (e < kTB * NR) Y[e / NR][e % NR] = make_float2(sign * v[i].x, sign * v[i].y);
      }
    };
    bool stop = false;
    fetch(0);
    for (int64_t jj = 0; jj < far; ++jj) {
      poll(jj);
      __syncthreads();  // every thread is done with the tiles of the previous block
      stop = s_abort;   // (set before this barrier only, so all threads agree)
      if (stop) break;
      store_tile();
      store_y(sm.Y[0], 1.f);
      fetch(jj + 1);  // in flight during the product below
      __syncthreads();
      stream_tile_product<NR>(sm.L, sm.Y[0], g, q, acc0, acc1);
    }
    if (stop) {  // every later wait gives up at once; this task stays unpublished
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      continue;
    }
    // right-hand side of the diagonal block: r = x - sum L_ij y_j, then D r
    stream_reduce<NR>(acc0, acc1, q);
    __syncthreads();  // every thread is done with the last factor tile
    stream_each<NR>(acc0, acc1, g, q, [&](int row, int k, float2 a) {
      float2 r = make_float2(0.f, 0.f);
      if (row < rows && k < nc) {
        const float2 xv = __ldg(x + (r0 + row) * ldx + k0 + k);
        r = make_float2(xv.x - a.x, xv.y - a.y);
      }
      sm.Y[0][row][k] = r;
    });
    store_tile();
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NR; ++k) acc0[k] = acc1[k] = make_float2(0.f, 0.f);
    stream_tile_product<NR>(sm.L, sm.Y[0], g, q, acc0, acc1);
    if (far < b) {  // - E_i y_h
      poll(far);
      store_y(sm.Y[1], -1.f);
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      if (s_abort) continue;
      stream_tile_product<NR>(sm.E, sm.Y[1], g, q, acc0, acc1);
    }
    stream_reduce<NR>(acc0, acc1, q);
    stream_each<NR>(acc0, acc1, g, q, [&](int row, int k, float2 a) {
      if (row < rows && k < nc) st_relaxed(y + (r0 + row) * ldx + k0 + k, a);
    });
  }
}

}  // namespace

// Blocks per superblock, and when a sweep uses them: one kernel takes nblk^2/2 tile products per
// chunk of columns, so with many right-hand sides sweeps change over to superblocks of 25 to 45 us
// (their own blocks) and 50 us per wave of update tiles.  One kernel / superblocks, ms per sweep:
// 15360 x 64 (nblk ceil(nrhs / 16) = 960) 2.26 / 2.40, 1920 x 642 (1230) 0.39 / 0.36, 7503 x 163 (1298)
// 1.43 / 1.25, 15360 x 163 (2640) 5.35 / 3.12, 7503 x 642 4.77 / 2.07, 15360 x 642 20.0 / 5.98.
constexpr int64_t kSuper = 8;
static bool use_superblocks(int64_t nblk, int64_t nrhs) { return nblk > kSuper && nblk * ((nrhs + 15) / 16) > 1100; }

// Columns per chunk.  The chain of a chunk takes 2.2 us per block with 4 columns, 3.2 with 8, 5.5 with
// 16, and the chunks run side by side until the tile products of all of them fill the SMs, about where
// 4 columns need 1200 block-chunks (ms per sweep with 4 / 8 / 16 columns: 1920 x 16 0.074 / 0.102 /
// 0.170, 1920 x 163 (1230) 0.157 / 0.164 / 0.235, 7503 x 16 0.278 / 0.404 / 0.663, 7503 x 64 (1888) 0.734 /
// 0.644 / 0.895, 15360 x 16 (960) 0.82 / 0.88 / 1.41, 15360 x 32 (1920) 1.48 / 1.29 / 1.84).
static int chunk_width(int64_t blocks, int64_t nrhs) {
  if (nrhs <= 2) return int(nrhs);
  return blocks * ((nrhs + 3) / 4) <= 1200 ? 4 : 8;
}

cudaError_t tri_block_inverses_c64(const void* LU, int64_t n, int64_t ld, void* Dinv, bool direct, cudaStream_t s) {
  const int64_t nblk = (n + kTB - 1) / kTB;
  if (nblk <= 0) return cudaSuccess;
  constexpr size_t kSmem = size_t(2) * kTB * (kTB + 1) * sizeof(float2);
  static bool attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr[dev]) {
    cudaError_t e = cudaFuncSetAttribute(tri_neighbour_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmem));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(tri_refine_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmem / 2 * 3));
    if (e != cudaSuccess) return e;
    attr[dev] = true;
  }
  const float2* lu = static_cast<const float2*>(LU);
  float2* d = static_cast<float2*>(Dinv);
  const int64_t one = nblk * kTB * kTB;
  for (int which = 0; which < 2; ++which) {
    tri_block_inverse_kernel<<<unsigned(nblk), 256, 0, s>>>(lu, n, ld, which, d + which * one);
    if (direct) tri_refine_kernel<<<unsigned(nblk), 256, kSmem / 2 * 3, s>>>(lu, n, ld, which, d + which * one);
    else tri_neighbour_kernel<<<unsigned(nblk), 256, kSmem, s>>>(lu, n, ld, which, d + which * one, d + (2 + which) * one);
  }
  return launched(4);
}

size_t tri_block_inverses_bytes(int64_t n) { return size_t(4 * ((n + kTB - 1) / kTB)) * kTB * kTB * sizeof(float2); }

size_t trsv_stream_tickets(int64_t n) { return size_t(((n + kTB - 1) / kTB + kSuper - 1) / kSuper); }

cudaError_t trsv_stream_c64(const void* LU, int64_t n, int64_t ld, const void* Dinv, void* X, void* Y, int64_t nrhs,
                            int64_t ldx, int upper, bool direct, int* tickets, int* status, cudaStream_t s) {
  if (n <= 0 || nrhs <= 0) return cudaSuccess;
  static int nsm[64] = {};
  static bool attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  cudaError_t e = cudaSuccess;
  if (!attr[dev]) {
    auto opt = [&](auto kern, size_t smem) {
      if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    };
    opt(trsv_stream_kernel<1>, sizeof(StreamSmem<1>));
    opt(trsv_stream_kernel<2>, sizeof(StreamSmem<2>));
    opt(trsv_stream_kernel<4>, sizeof(StreamSmem<4>));
    opt(trsv_stream_kernel<8>, sizeof(StreamSmem<8>));
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    attr[dev] = true;
  }
  const int64_t nblk = (n + kTB - 1) / kTB, one = nblk * kTB * kTB;
  const bool super = use_superblocks(nblk, nrhs);
  const int64_t step = super ? kSuper : nblk;
  const int w = chunk_width(step, nrhs);
  const int64_t chunks = (nrhs + w - 1) / w;
  e = cudaMemsetAsync(tickets, 0, sizeof(int) * trsv_stream_tickets(n), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(Y, 0xFF, sizeof(float2) * size_t(n) * size_t(ldx), s);  // nothing ready
  if (e != cudaSuccess) return e;
  const float2* L = static_cast<const float2*>(LU);
  const float2* D = static_cast<const float2*>(Dinv) + (upper ? one : 0);
  const float2* E = static_cast<const float2*>(Dinv) + (upper ? 3 : 2) * one;
  float2* x = static_cast<float2*>(X);
  float2* y = static_cast<float2*>(Y);
  for (int64_t first = 0, q = 0; first < nblk; first += step, ++q) {
    const int64_t count = std::min(step, nblk - first);
    const unsigned grid = unsigned(std::min<int64_t>(count * chunks, int64_t(2) * std::max(nsm[dev], 1)));
    auto run = [&](auto kern, size_t smem) -> cudaError_t {
      kern<<<grid, 256, smem, s>>>(L, n, ld, D, E, x, y, nrhs, ldx, chunks, first, count, upper, direct ? 0 : 1, tickets + q, status);
      return launched();
    };
    switch (w) {
      case 1: e = run(trsv_stream_kernel<1>, sizeof(StreamSmem<1>)); break;
      case 2: e = run(trsv_stream_kernel<2>, sizeof(StreamSmem<2>)); break;
      case 4: e = run(trsv_stream_kernel<4>, sizeof(StreamSmem<4>)); break;
      default: e = run(trsv_stream_kernel<8>, sizeof(StreamSmem<8>)); break;
    }
    if (e != cudaSuccess) return e;
    if (first + count == nblk) break;
    // rows [lo, hi) are solved: take them out of the rows that follow in the sweep
    const int64_t lo = upper ? (nblk - first - count) * kTB : first * kTB;
    const int64_t hi = upper ? std::min(n, (nblk - first) * kTB) : (first + count) * kTB;
    const int64_t r0 = upper ? 0 : hi, r1 = upper ? lo : n;
    e = cgemm_update_tc(r1 - r0, nrhs, hi - lo, L + r0 * ld + lo, ld, y + lo * ldx, ldx, x + r0 * ldx, ldx, status, s,
                        "trsm_update");
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Sets the poll limit of the sweep flag waits on the current device (polls <= 0: the default).
cudaError_t set_wait_limit_sweeps(long long polls) {
  const long long v = polls > 0 ? polls : kFlagSpinLimit;
  return cudaMemcpyToSymbol(g_flag_wait_limit, &v, sizeof(v));
}

}  // namespace fosb
