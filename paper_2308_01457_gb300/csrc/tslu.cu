// Tournament-pivoting panel factorisation (TSLU) of a complex64 m x jb panel (jb <= 64),
// for the blocked LU of the mixed and FP32 paths.
//
// Partial pivoting needs one grid-wide reduction per column.  Here the pivot rows of the
// whole panel are chosen by a reduction tree instead:
//   1. leaves: every cluster of CTAs factors a block of up to 2048 rows with partial pivoting
//      and nominates the rows it pivoted on (at most jb);
//   2. tree: a cluster merges up to 32 nominee sets (<= 2048 rows, original values re-read from
//      the panel) the same way until one set of jb rows remains (up to 2048 rows: one level, up
//      to 65,536: two); its factorisation is L11 \ U11 of the panel in the chosen pivot order;
//   3. the last cluster also writes L11 \ U11 into the top jb rows, moves the displaced rows and
//      lists the row moves for the other columns;
//   4. L21 = A21 U11^{-1}, four threads per row.
// The panel stays untouched in global memory until step 3, so every level reads original
// rows.  Launches are stream-ordered; CTAs wait for one another inside a cluster only.
//
// Within a cluster the candidate rows sit in the CTAs' shared memory (up to 256 each) and are
// factored by blocked partial pivoting in blocks of 8 columns (panel_cluster_kernel).  This is
// unblocked partial pivoting whose pivot magnitudes are compared on 15 mantissa bits (a
// candidate within a relative 2^-15 of the largest may win the tie, so |l| <= 1 + 2^-15).
// Rows are never moved: a row that has served as pivot is marked used, keeps its (L, U)
// entries and is skipped by later updates, so at the end the row chosen at step j holds row j
// of L \ U.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>
#include <type_traits>

#include "fosb_internal.h"

namespace fosb {
namespace {

constexpr int kTsluCols = 64;      // panel width handled (jb <= 64)
constexpr int kTsluBlk = 8;        // columns per block of the blocked factorisation
constexpr int kTsluThreads = 512;
constexpr int kTsluCluster = 8;    // CTAs per cluster (one for panels of at most 256 rows)
constexpr int kTsluMaxRows = 256;  // rows per CTA
constexpr long long kTsluSpin = 1ll << 25;

__device__ __forceinline__ float2 cinv(float2 v) {
  const float den = v.x * v.x + v.y * v.y;
  if (!(den > 0.f)) return make_float2(0.f, 0.f);
  const float r = __frcp_rn(den);
  return make_float2(v.x * r, -v.y * r);
}
__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ void cfms(float2& a, float2 l, float2 u) {  // a -= l u
  a.x = fmaf(l.y, u.y, fmaf(-l.x, u.x, a.x));
  a.y = fmaf(-l.y, u.x, fmaf(-l.x, u.y, a.y));
}
__device__ __forceinline__ void cfms2(float4& a, float2 l, float4 u) {  // both complex values of a pair
  a.x = fmaf(l.y, u.y, fmaf(-l.x, u.x, a.x));
  a.y = fmaf(-l.y, u.x, fmaf(-l.x, u.y, a.y));
  a.z = fmaf(l.y, u.w, fmaf(-l.x, u.z, a.z));
  a.w = fmaf(-l.y, u.z, fmaf(-l.x, u.w, a.w));
}

// ---- cluster and mbarrier pieces (shared-window addresses)
__device__ __forceinline__ uint32_t sptr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
// 16 bytes into a CTA of the cluster, counted on that CTA's mbarrier
__device__ __forceinline__ void push16(uint32_t dst, float4 v, uint32_t mbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst),
               "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)),
               "r"(__float_as_uint(v.w)), "r"(mbar)
               : "memory");
}
__device__ __forceinline__ void expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(mbar), "r"(bytes)
               : "memory");
}
// Bounded wait for a phase of a local mbarrier; false once it gives up or another wait has.
__device__ __forceinline__ bool phase_wait(uint32_t mbar, uint32_t parity, volatile int* stop) {
  for (long long i = 0; i < kTsluSpin; ++i) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) return true;
    if ((i & 1023) == 1023 && *stop) return false;
  }
  return false;
}

__device__ __forceinline__ void step_bar(int n) { asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory"); }

// A pivot candidate: the row's block columns from the step's on, the inverse of its pivot value
// and its key.
struct Cand {
  float4 row[kTsluBlk / 2];
  float2 inv;
  unsigned key, pad;
};
static_assert(sizeof(Cand) == 80, "a candidate is five 16-byte pushes");

// Shared memory of a CTA with ROWS candidate rows.  In the block update a warp covers 4 rows x 8
// column pairs, so an 8-thread access phase is 128 contiguous bytes of one row; the row pitch
// (34 16-byte units) spreads the pivot steps' column accesses over the banks.
template <int ROWS>
struct PanelSmem {
  static constexpr int LD = 68;         // complex values
  static constexpr int LU = 66;         // of a row of U: the column solve reads 8 rows x 4 columns
  static constexpr int AW = ROWS / 32;  // warps that own rows
  float2 A[ROWS][LD];
  // The CTAs' candidates of the eight steps of a block.  A peer can be one step ahead, and its
  // push for the first step of a block needs nothing of this CTA's block end, so that step
  // alternates slots.
  Cand cand[kTsluBlk + 1][kTsluCluster];
  Cand stage[2][AW];              // the warps' candidates, by step parity
  float2 U[kTsluBlk][LU];         // the block's pivot rows from the block on, then U12 right of it
  int rows[ROWS];
  int own[kTsluCols];  // row of this CTA chosen at each step, or -1
  int win[kTsluBlk];   // winning CTA of each step of the block | row << 16
  int sel[kTsluCols], disp[kTsluCols], vac[kTsluCols], flag[kTsluCols];  // last level: the row moves
  unsigned mask[2][2];
  unsigned char used[ROWS];
  uint64_t bar_step[kTsluBlk], bar_u;
  int stop, ndisp;
};

// One level of the tree.  Leaf mode (in_idx == nullptr): cluster b holds panel rows
// [b * rows_per, min(m, (b + 1) * rows_per)).  Tree mode: cluster b holds the nominees of groups
// [b * fan, min(groups_in, (b + 1) * fan)), group g's panel rows at in_idx[g * 64 ...] (64 of them, but for the
// last group in_last).  The rows are split evenly over the cluster's CTAs.  Every cluster writes
// its pivot rows in order to out_idx[b * 64 ...] and the last cluster's count to out_last.  A
// launch of one cluster is the root: it finishes the panel (step 3 above).
//
// A pivot step of an 8-column block runs on the warps that own rows, a thread per row with the
// row's eight block columns in registers: a warp argmax (one redux.sync of a 32-bit key), a
// barrier among these warps, an argmax over the warps' staged candidates, the CTA's candidate
// pushed into every CTA of the cluster by its warp (st.async, counted by the receivers'
// mbarriers), an argmax over the CTAs' and the elimination of the column inside the block.  One
// push per CTA, not per warp: 64 candidates per step bound the cluster's traffic (700 clocks a
// step against 300).  No cluster barrier is on that path: its length is the one-way push.
// Warp 8 + j watches step j of the block, and where its CTA owns the pivot row pushes the row
// (its multipliers inside the block and its trailing columns) to all CTAs; at the block's end each
// CTA forms U12 = L11^{-1} A12 from them, eight lanes per column, and updates its own rows by all
// sixteen warps.  A lone CTA (CL = 1) pushes nothing.  The steps are one rolled loop on a register
// window that shifts by a column per step (unrolled, a level over 1000 rows took 58.7 us, rolled
// 52.6).  Latency-bound: about 1000 clocks per step, 300 of them the push, and 3000 to 6000 per
// block update (128 or 256 rows).  A panel of 1000 rows takes 53 us, one of 15360 rows about 100
// us; one CTA per 256 rows with fan-in 4 took 53 us for each of 3 (4) levels and 10 us for step 3.
template <int ROWS, int CL>
__global__ void __launch_bounds__(kTsluThreads, 1)
    panel_cluster_kernel(float2* __restrict__ A, int64_t lda, int64_t m, int jb, int64_t rows_per,
                         const int* __restrict__ in_idx, int groups_in, int fan, const int* __restrict__ in_last,
                         int* __restrict__ out_idx, int* __restrict__ out_last, int* __restrict__ sel,
                         int2* __restrict__ moves, int* __restrict__ status) {
  using S = PanelSmem<ROWS>;
  constexpr int AW = S::AW;
  extern __shared__ __align__(16) unsigned char panel_raw[];
  S& sm = *reinterpret_cast<S*>(panel_raw);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  uint32_t rank_u;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank_u));
  const int rank = int(rank_u), cluster = int(blockIdx.x) / CL;
  const bool root = int(gridDim.x) == CL;
  // this cluster's candidate rows, and this CTA's share of them
  int total;
  if (in_idx == nullptr) {
    const int64_t lo = int64_t(cluster) * rows_per;
    total = int(min(rows_per, m - lo));
  } else {
    const int g0 = cluster * fan, g1 = min(groups_in, g0 + fan);
    total = (g1 - g0) * kTsluCols;
    if (g1 == groups_in) total -= kTsluCols - *in_last;
  }
  const int per = (total + CL - 1) / CL, first = rank * per, nr = max(0, min(per, total - first));
  if (t < ROWS) {
    int row = 0;
    if (t < nr) row = in_idx == nullptr ? int(int64_t(cluster) * rows_per) + first + t
                                        : in_idx[int64_t(cluster) * fan * kTsluCols + first + t];
    sm.rows[t] = row;
    sm.used[t] = t >= nr;
  }
  if (t < kTsluCols) sm.own[t] = -1;
  if (t == 0) {
    for (int i = 0; i < kTsluBlk; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sptr(&sm.bar_step[i])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sptr(&sm.bar_u)));
    asm volatile("fence.mbarrier_init.release.cluster;");
    sm.stop = 0;
  }
  __syncthreads();
  const int steps = min(total, jb);
  // rows into shared memory, a warp per row (256 contiguous bytes per load instruction), all of a
  // warp's loads in flight; zero past jb and for missing rows
  {
    constexpr int kWarps = kTsluThreads / 32, kBatch = ROWS / kWarps;
    float2 v[kBatch][2];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int rr = warp + b * kWarps;
      const float2* src = A + int64_t(sm.rows[rr]) * lda;
      v[b][0] = (rr < nr && lane < jb) ? src[lane] : make_float2(0.f, 0.f);
      v[b][1] = (rr < nr && lane + 32 < jb) ? src[lane + 32] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int rr = warp + b * kWarps;
      sm.A[rr][lane] = v[b][0];
      sm.A[rr][lane + 32] = v[b][1];
    }
  }
  // valid rows in every output first: if a wait gives up, the steps not reached keep them
  if (rank == 0 && t < kTsluCols) {
    if (root) sel[t] = t < jb ? t : 0;
    else out_idx[int64_t(cluster) * kTsluCols + t] = sm.rows[min(t, nr - 1)];
  }
  cluster_sync();  // rows in shared memory, mbarriers ready in every CTA
  auto give_up = [&]() {
    *static_cast<volatile int*>(&sm.stop) = 1;
    atomicExch(status, FOSB_ERR_TIMEOUT);
  };
  // the largest of n candidates' keys (equal keys: the lowest index): its index
  auto winner = [&](const Cand* c, int n, unsigned& key) -> int {
    const unsigned k = lane < n ? c[lane].key : 0u;
    key = __reduce_max_sync(0xffffffffu, k);
    return __ffs(__ballot_sync(0xffffffffu, lane < n && k == key)) - 1;
  };
  bool used = t >= nr;  // (row threads: warps below AW)
  int order = -1;
  const int npairs = (jb + 1) >> 1;
#pragma unroll 1
  for (int cb = 0, blk = 0; cb < steps; cb += kTsluBlk, ++blk) {
    const uint32_t par = blk & 1;
    const int ce = min(cb + kTsluBlk, steps), npiv = ce - cb;  // pivot steps of this block
    const bool more = ce < steps;                              // then npiv = 8 and a block follows
    const int width = kTsluCols - cb;                          // columns from the block on (padded panel)
    const int bar_n = 32 * (AW + (CL > 1 && more ? 1 : 0));    // the row warps and the step's watcher
    if (CL > 1 && t == 0) {
      for (int i = 0; i < npiv; ++i) expect_tx(sptr(&sm.bar_step[i]), uint32_t(CL * sizeof(Cand)));
      if (more) expect_tx(sptr(&sm.bar_u), uint32_t(npiv * width * sizeof(float2)));
    }
    if (warp < AW) {
      float2 bv[kTsluBlk];  // the row's block columns from the current step's on
      const float4* myb = reinterpret_cast<const float4*>(&sm.A[t][cb]);
#pragma unroll
      for (int i = 0; i < kTsluBlk / 2; ++i) {
        const float4 w = myb[i];
        bv[2 * i] = make_float2(w.x, w.y);
        bv[2 * i + 1] = make_float2(w.z, w.w);
      }
#pragma unroll 1
      for (int jj = 0; jj < npiv; ++jj) {
        // pivot: the largest |Re| + |Im| in the column among unused rows, compared on the top
        // 24 bits of its float pattern (15 mantissa bits).  One 32-bit key per row: bit 31
        // marks a candidate, the low 8 bits hold 255 - row.
        const float2 vj = bv[0];
        const unsigned key =
            used ? 0u
                 : (0x80000000u | (__float_as_uint(fabsf(vj.x) + fabsf(vj.y)) & 0x7FFFFF00u) | unsigned(255 - t));
        const float2 myinv = cinv(vj);  // the inverse as pivot, ready before the argmax ends
        const unsigned mk = __reduce_max_sync(0xffffffffu, key);
        Cand* stage = sm.stage[jj & 1];
        if (key == mk && (mk != 0u || lane == 0)) {  // this warp's candidate (the row bits make it unique)
          Cand& st = stage[warp];
          st.key = mk;
          st.inv = myinv;
#pragma unroll
          for (int i = 0; i < kTsluBlk / 2; ++i)
            st.row[i] = make_float4(bv[2 * i].x, bv[2 * i].y, bv[2 * i + 1].x, bv[2 * i + 1].y);
        }
        step_bar(bar_n);
        unsigned g = __reduce_max_sync(0xffffffffu, lane < AW ? stage[lane].key : 0u);
        const int lw = (int(255u - (g & 255u)) & (ROWS - 1)) >> 5;  // the row bits name the warp
        const Cand* best = stage + lw;
        int wr = 0;
        if constexpr (CL > 1) {
          Cand* slots = sm.cand[jj == 0 && par ? kTsluBlk : jj];
          const uint32_t bar = sptr(&sm.bar_step[jj]);
          if (warp == lw) {
            const float4* src = reinterpret_cast<const float4*>(best);
            const uint32_t dst = sptr(&slots[rank]);
            const int part = lane & 3, d = lane >> 2;
            const float4 a = src[part], b = src[4];
            if (d < CL) push16(map_rank(dst + 16 * part, d), a, map_rank(bar, d));
            if (lane < CL) push16(map_rank(dst + 64, lane), b, map_rank(bar, lane));
          }
          if (!phase_wait(bar, par, &sm.stop)) give_up();
          wr = winner(slots, CL, g);
          best = slots + wr;
        }
        const int p = int(255u - (g & 255u)) & (ROWS - 1);
        if (wr == rank && t == p) {
          used = true;
          order = cb + jj;
        }
        if (!used) {  // eliminate the column from my block columns and move on by one
          const float2 l = cmulf(vj, best->inv);
          float2 r[kTsluBlk];
#pragma unroll
          for (int i = 0; i < kTsluBlk / 2; ++i) {
            const float4 w = best->row[i];
            r[2 * i] = make_float2(w.x, w.y);
            r[2 * i + 1] = make_float2(w.z, w.w);
          }
#pragma unroll
          for (int i = 1; i < kTsluBlk; ++i) {
            bv[i - 1] = bv[i];
            cfms(bv[i - 1], l, r[i]);
          }
          bv[kTsluBlk - 1] = make_float2(0.f, 0.f);
          sm.A[t][cb + jj] = l;
        }
        if (t == 0) sm.win[jj] = wr | (p << 16);
      }
      if (order >= cb) {  // chosen in this block: its row of U inside the block
        sm.used[t] = 1;
        sm.own[order] = t;
#pragma unroll
        for (int i = 0; i < kTsluBlk; ++i)
          if (order + i < cb + kTsluBlk) sm.A[t][order + i] = bv[i];
      }
    } else if (CL > 1 && warp >= 8 && more) {
      // the watcher of step jj: once the step before it is decided it meets the row warps (whose
      // multipliers it then sees), and where this CTA owns the pivot row it pushes the row
      const int jj = warp - 8;
      bool ok = jj == 0 || phase_wait(sptr(&sm.bar_step[jj - 1]), par, &sm.stop);
      step_bar(bar_n);
      ok = ok && phase_wait(sptr(&sm.bar_step[jj]), par, &sm.stop);
      if (!ok) give_up();
      unsigned g;
      if (winner(sm.cand[jj == 0 && par ? kTsluBlk : jj], CL, g) == rank) {
        const int p = int(255u - (g & 255u)) & (ROWS - 1);
        const uint32_t bar = sptr(&sm.bar_u);
        if (lane < width / 2) {
          const float4 v = reinterpret_cast<const float4*>(&sm.A[p][cb])[lane];
          const uint32_t dst = sptr(&sm.U[jj][cb]) + 16 * lane;
          for (int d = 0; d < CL; ++d) push16(map_rank(dst, d), v, map_rank(bar, d));
        }
      }
    }
    __syncthreads();  // block columns, win and used are in shared memory
    if (!more) break;  // the same for every thread of the cluster
    // U12 = L11^{-1} A12 (L11 unit lower, the pivot rows' multipliers inside the block): lane (c, i)
    // of a column's eight holds row i's entry; the owner keeps it as its row of U
    if (t < kTsluBlk * (kTsluCols - kTsluBlk)) {
      const int i = t & 7, c = cb + kTsluBlk + (t >> 3);
      if (CL > 1 && !phase_wait(sptr(&sm.bar_u), par, &sm.stop)) give_up();
      const int w = sm.win[i];
      const float2* row = CL > 1 ? sm.U[i] : sm.A[w >> 16];
      float2 u = c < kTsluCols ? row[c] : make_float2(0.f, 0.f);
#pragma unroll
      for (int q = 0; q < kTsluBlk - 1; ++q) {
        const float2 l = row[cb + q];
        const float2 x = make_float2(__shfl_sync(0xffffffffu, u.x, q, 8), __shfl_sync(0xffffffffu, u.y, q, 8));
        if (i > q) cfms(u, l, x);
      }
      if (c < kTsluCols) {
        sm.U[i][c] = u;
        if ((w & 0xffff) == rank) sm.A[w >> 16][c] = u;
      }
    }
    __syncthreads();
    if (sm.stop) break;  // a wait gave up: the same for every thread of this CTA
    // rank-8 update of the rows not chosen yet over their column pairs right of the block: thread
    // (r, h) takes rows r, r + 64, ... two at a time (each value of U read once for both) and the
    // pairs P with P % 8 == h
    {
      const int r0 = t >> 3, h = t & 7;
      const float4* u = reinterpret_cast<const float4*>(sm.U);
      constexpr int kRow = S::LU / 2;  // float4 per row of U
#pragma unroll 1
      for (int q = 0; q < ROWS / 128; ++q) {
        const int ra = r0 + 128 * q, rb = ra + 64;
        const bool ua = !sm.used[ra], ub = !sm.used[rb];
        if (ua || ub) {
          float4* pa = reinterpret_cast<float4*>(sm.A[ra]);
          float4* pb = reinterpret_cast<float4*>(sm.A[rb]);
          float2 la[kTsluBlk], lb[kTsluBlk];
#pragma unroll
          for (int i = 0; i < kTsluBlk; i += 2) {
            const float4 v = pa[(cb + i) >> 1], w = pb[(cb + i) >> 1];
            la[i] = make_float2(v.x, v.y);
            la[i + 1] = make_float2(v.z, v.w);
            lb[i] = make_float2(w.x, w.y);
            lb[i + 1] = make_float2(w.z, w.w);
          }
#pragma unroll 1
          for (int P = ((cb + kTsluBlk) >> 1) + h; P < npairs; P += 8) {
            float4 a = pa[P], b = pb[P];
#pragma unroll
            for (int i = 0; i < kTsluBlk; ++i) {
              const float4 uu = u[i * kRow + P];
              cfms2(a, la[i], uu);
              cfms2(b, lb[i], uu);
            }
            if (ua) pa[P] = a;
            if (ub) pb[P] = b;
          }
        }
      }
    }
    __syncthreads();
  }
  if (!root) {
    if (order >= 0) out_idx[int64_t(cluster) * kTsluCols + order] = sm.rows[t];
    if (t == 0 && rank == 0 && cluster == int(gridDim.x) / CL - 1) *out_last = steps;
    if (sm.stop) __nanosleep(20000);  // pushes of a peer that gave up may still be on their way
    cluster_sync();
    return;
  }
  if (sm.stop) __nanosleep(20000);  // pushes of a peer that gave up may still be on their way
  // ---- root: position i receives row sel[i]; the top rows that were not chosen go, in order, to
  // the positions the chosen rows leave below the top
  if (order >= 0) sel[order] = sm.rows[t];
  cluster_sync();
  if (t < kTsluCols) {
    sm.sel[t] = t < jb ? __ldcg(sel + t) : -1;
    sm.flag[t] = 0;
  }
  __syncthreads();
  if (t < jb && sm.sel[t] >= 0 && sm.sel[t] < jb) sm.flag[sm.sel[t]] = 1;
  __syncthreads();
  // ranks among the displaced top rows and among the vacated positions
  const bool out = t < jb && !sm.flag[t & (kTsluCols - 1)], hole = t < jb && sm.sel[t & (kTsluCols - 1)] >= jb;
  if (warp < 2) {
    const unsigned mo = __ballot_sync(0xffffffffu, out), mh = __ballot_sync(0xffffffffu, hole);
    if (lane == 0) {
      sm.mask[0][warp] = mo;
      sm.mask[1][warp] = mh;
    }
  }
  __syncthreads();
  if (warp < 2) {
    const unsigned below = (1u << lane) - 1u;
    const int nd = __popc(sm.mask[0][warp] & below) + (warp ? __popc(sm.mask[0][0]) : 0);
    const int nv = __popc(sm.mask[1][warp] & below) + (warp ? __popc(sm.mask[1][0]) : 0);
    if (out) sm.disp[nd] = t;
    if (hole) sm.vac[nv] = sm.sel[t];
    if (t == 0)
      sm.ndisp = min(__popc(sm.mask[0][0]) + __popc(sm.mask[0][1]), __popc(sm.mask[1][0]) + __popc(sm.mask[1][1]));
  }
  __syncthreads();
  const int ndisp = sm.ndisp;
  constexpr int kPer = kTsluCols / (kTsluThreads / 32);
  float2 keep[kPer][2];
  if (rank == 0) {
    if (t < jb) {
      const int s = sm.sel[t];
      moves[t] = s != t && s >= 0 && s < m ? make_int2(s, t) : make_int2(-1, -1);
      moves[jb + t] = t < ndisp && sm.vac[t] < m ? make_int2(sm.disp[t], sm.vac[t]) : make_int2(-1, -1);
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) {  // the displaced rows' panel columns
      const int i = warp + q * (kTsluThreads / 32);
      const float2* src = A + int64_t(i < ndisp ? sm.disp[i] : 0) * lda;
      keep[q][0] = (i < ndisp && lane < jb) ? src[lane] : make_float2(0.f, 0.f);
      keep[q][1] = (i < ndisp && lane + 32 < jb) ? src[lane + 32] : make_float2(0.f, 0.f);
    }
  }
  cluster_sync();  // every top row that moves has been read
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int i = warp + q * (kTsluThreads / 32);
    if (rank == 0 && i < ndisp && sm.vac[i] < m) {
      float2* dst = A + int64_t(sm.vac[i]) * lda;
      if (lane < jb) dst[lane] = keep[q][0];
      if (lane + 32 < jb) dst[lane + 32] = keep[q][1];
    }
    const int p = i < jb ? sm.own[i] : -1;
    if (p >= 0) {  // L11 \ U11, row i
      float2* dst = A + int64_t(i) * lda;
      if (lane < jb) dst[lane] = sm.A[p][lane];
      if (lane + 32 < jb) dst[lane + 32] = sm.A[p][lane + 32];
      const float2 d = sm.A[p][i];
      if (lane == 0 && !(d.x != 0.f || d.y != 0.f)) atomicCAS(status, 0, FOSB_ERR_SINGULAR);
    }
  }
}

// Triangular substitution on vectors of 64 complex values, four threads per vector: thread h
// holds elements 16 h .. 16 h + 15 in registers.  For k = 0 .. 63, x_k *= dinv_k (kScale) and
// x_c -= x_k M[k][c] for c > k, the right-looking order of forward substitution: 8 elements at a
// time are solved by the thread that holds them and published (s_x, by the parity of the chunk: one
// barrier per chunk), then one rank-8 update reaches every later element (the same operations in
// the same order as one element at a time).  M is in shared memory and read by every thread of a
// warp alike.  Bound by the shared-memory reads of M (one 16-byte read per 8 FMAs) and the chain of
// 8 chunks: 13.3 us for L21 (rows) and 10.8 us for U12 (columns) per panel, 25.7 and 20.7 us with a thread
// per vector, which ran 2016 dependent complex steps.
constexpr int kTriVec = 64;                   // vectors per CTA
constexpr int kTriThreads = 4 * kTriVec;
constexpr int kTriLd = kTriVec + 1;
template <bool kScale>
__device__ __forceinline__ void tri_quad(float2 (&y)[16], int h, int v, const float2 (*M)[kTsluCols],
                                         const float2* dinv, float2 (*s_x)[8][kTriVec]) {
#pragma unroll 1
  for (int q = 0; q < 4; ++q) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int k0 = 16 * q + 8 * half, b = 8 * half;
      if (h == q) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (kScale) y[b + i] = cmulf(y[b + i], dinv[k0 + i]);
          s_x[half][i][v] = y[b + i];
#pragma unroll
          for (int p = i + 1; p < 8; ++p) cfms(y[b + p], y[b + i], M[k0 + i][k0 + p]);
        }
      }
      __syncthreads();
      if (h < q || (h == q && half == 1)) continue;  // nothing later in this thread
      float2 x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = s_x[half][i][v];
      const float4* m4 = reinterpret_cast<const float4*>(&M[k0][16 * h]);
#pragma unroll
      for (int c = 0; c < 16; c += 2) {
        if (c < 8 && h == q) continue;  // (half 0) the chunk itself
        float4 a = make_float4(y[c].x, y[c].y, y[c + 1].x, y[c + 1].y);
#pragma unroll
        for (int i = 0; i < 8; ++i) cfms2(a, x[i], m4[i * (kTsluCols / 2) + c / 2]);
        y[c] = make_float2(a.x, a.y);
        y[c + 1] = make_float2(a.z, a.w);
      }
    }
  }
}

struct LsSmem {
  float2 M[kTsluCols][kTsluCols];
  float2 xs[kTsluCols][kTriLd];
  float2 x[2][8][kTriVec];
  float2 dinv[kTsluCols];
};
constexpr size_t kLsSmem = sizeof(LsSmem);

// L21 = A21 U11^{-1} for rows [jb, m), U11 the upper triangle (with the diagonal) of the top
// jb rows.  The CTA's 64 rows are loaded with coalesced row reads, 8 rows in flight per warp, into
// a transposed shared tile; U11 is staged identity-padded to 64 x 64, so a ragged panel
// (jb < 64) needs no other case.
__global__ void __launch_bounds__(kTriThreads) tslu_lsolve_kernel(float2* __restrict__ A, int64_t lda, int64_t m,
                                                                  int jb) {
  extern __shared__ float4 ls_raw[];
  LsSmem& sm = *reinterpret_cast<LsSmem*>(ls_raw);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  constexpr int kWarps = kTriThreads / 32, kBatch = kTriVec / kWarps;
  for (int e = t; e < kTsluCols * kTsluCols; e += kTriThreads) {
    const int r = e / kTsluCols, c = e % kTsluCols;
    sm.M[r][c] = (r < jb && c < jb && c >= r) ? A[int64_t(r) * lda + c] : make_float2(0.f, 0.f);
  }
  const int64_t r0 = jb + int64_t(blockIdx.x) * kTriVec;
  {
    float2 v[kBatch][2];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int64_t row = r0 + warp + b * kWarps;
      v[b][0] = (row < m && lane < jb) ? A[row * lda + lane] : make_float2(0.f, 0.f);
      v[b][1] = (row < m && lane + 32 < jb) ? A[row * lda + lane + 32] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int rr = warp + b * kWarps;
      sm.xs[lane][rr] = v[b][0];
      sm.xs[lane + 32][rr] = v[b][1];
    }
  }
  __syncthreads();
  if (t < kTsluCols) sm.dinv[t] = t < jb ? cinv(sm.M[t][t]) : make_float2(1.f, 0.f);
  const int v = t & (kTriVec - 1), h = t / kTriVec;
  float2 y[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) y[i] = sm.xs[16 * h + i][v];
  __syncthreads();
  tri_quad<true>(y, h, v, sm.M, sm.dinv, sm.x);
#pragma unroll
  for (int i = 0; i < 16; ++i) sm.xs[16 * h + i][v] = y[i];
  __syncthreads();
#pragma unroll
  for (int b = 0; b < kBatch; ++b) {
    const int rr = warp + b * kWarps;
    const int64_t row = r0 + rr;
    if (row >= m) break;
    if (lane < jb) A[row * lda + lane] = sm.xs[lane][rr];
    if (lane + 32 < jb) A[row * lda + lane + 32] = sm.xs[lane + 32][rr];
  }
}

// X (jb x ncols, leading dimension ldx) := L^{-1} X with L the unit lower jb x jb block at
// D (leading dimension ldd): a vector per column, M[k][c] = L[c][k] staged zero-padded.
__global__ void __launch_bounds__(kTriThreads) tri_lower_unit_cols_kernel(const float2* __restrict__ D, int64_t ldd,
                                                                          int jb, float2* __restrict__ X, int64_t ldx,
                                                                          int64_t ncols) {
  __shared__ __align__(16) float2 sM[kTsluCols][kTsluCols];
  __shared__ float2 s_x[2][8][kTriVec];
  const int t = threadIdx.x, v = t & (kTriVec - 1), h = t / kTriVec;
  const int64_t col = int64_t(blockIdx.x) * kTriVec + v;
  float2 y[16];
#pragma unroll
  for (int i = 0; i < 16; ++i)
    y[i] = (col < ncols && 16 * h + i < jb) ? X[int64_t(16 * h + i) * ldx + col] : make_float2(0.f, 0.f);
  for (int e = t; e < kTsluCols * kTsluCols; e += kTriThreads) {
    const int c = e / kTsluCols, k = e % kTsluCols;  // (coalesced along a row of L)
    sM[k][c] = (k < jb && c < jb && c > k) ? D[int64_t(c) * ldd + k] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  tri_quad<false>(y, h, v, sM, nullptr, s_x);
  if (col >= ncols) return;
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (16 * h + i < jb) X[int64_t(16 * h + i) * ldx + col] = y[i];
}

// The panel's row permutation on the columns outside it (left: earlier L columns; right:
// the trailing matrix).  Row j0 + dst takes the old values of row j0 + src for every move
// (at most 2 jb rows, each a source once and a destination once), and so does the composed row
// permutation perm (block 0).  A CTA covers 32 columns: lanes run along a row (256-byte
// accesses), the 8 warps split the moves, and every read of the CTA's columns happens before any
// write.
__global__ void __launch_bounds__(256) tslu_swap_kernel(float2* __restrict__ A, int64_t n, int64_t lda, int64_t j0,
                                                        int jb, const int2* __restrict__ moves,
                                                        int32_t* __restrict__ perm) {
  __shared__ int2 s_mv[2 * kTsluCols];
  const int t = threadIdx.x;
  if (t < 2 * jb) s_mv[t] = moves[t];
  __syncthreads();
  int32_t moved = 0;
  const bool mine = blockIdx.x == 0 && t < 2 * jb && s_mv[t].x >= 0;
  if (mine) moved = perm[j0 + s_mv[t].x];
  const int tx = t & 31, ty = t >> 5;
  const int64_t c = int64_t(blockIdx.x) * 32 + tx;
  const bool col_ok = c < n && (c < j0 || c >= j0 + jb);
  constexpr int kPer = 2 * kTsluCols / 8;
  float2 v[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int mi = ty + 8 * k;
    if (col_ok && mi < 2 * jb && s_mv[mi].x >= 0) v[k] = A[(j0 + s_mv[mi].x) * lda + c];
  }
  __syncthreads();
  if (mine) perm[j0 + s_mv[t].y] = moved;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int mi = ty + 8 * k;
    if (col_ok && mi < 2 * jb && s_mv[mi].x >= 0) A[(j0 + s_mv[mi].y) * lda + c] = v[k];
  }
}

inline unsigned cdivu(int64_t a, int64_t b) { return unsigned((a + b - 1) / b); }

}  // namespace

namespace {

__global__ void iota_kernel(int32_t* p, int64_t n) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) p[i] = int32_t(i);
}

// Clusters of kTsluCluster CTAs that this device can hold at once (per rows-per-CTA variant), with
// the kernels' shared memory opted in; < 1 on an error.
int max_clusters(int rows) {
  static std::mutex mu;
  static int cached[64][2] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lock(mu);
  int& c = cached[dev][rows == 256];
  if (c > 0) return c;
  auto query = [&](auto kern, size_t smem) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kTsluCluster);
    cfg.blockDim = dim3(kTsluThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kTsluCluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    return cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess ? n : 0;
  };
  // the one-CTA variants take the same opt-in
  auto opt_in = [&](auto kern, size_t smem) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) == cudaSuccess;
  };
  if (!(rows == 256 ? opt_in(panel_cluster_kernel<256, 1>, sizeof(PanelSmem<256>))
                    : opt_in(panel_cluster_kernel<128, 1>, sizeof(PanelSmem<128>))))
    return 0;
  c = rows == 256 ? query(panel_cluster_kernel<256, kTsluCluster>, sizeof(PanelSmem<256>))
                  : query(panel_cluster_kernel<128, kTsluCluster>, sizeof(PanelSmem<128>));
  return c;
}

// Rows per CTA and number of clusters of a level over `rows` rows.  Up to 256 rows one CTA holds
// everything (no push leaves it); else clusters of eight, with 128 rows per CTA (half the block
// update per step of a level) where the level then needs no more clusters than fit at once and no
// more levels, else 256.
struct Level {
  int rows_per_cta, cl, clusters;
};
Level plan_level(int64_t rows) {
  if (rows <= kTsluMaxRows) return {rows <= 128 ? 128 : 256, 1, 1};
  const int64_t half = (rows + 1023) / 1024, full = (rows + 2047) / 2048;
  if (half == 1 || (full > 1 && half <= std::min(16, max_clusters(128)))) return {128, kTsluCluster, int(half)};
  return {256, kTsluCluster, int(full)};
}

}  // namespace

size_t tslu_scratch_bytes(int64_t n) {
  const int64_t groups = std::max<int64_t>((n + 2047) / 2048, 16);
  return size_t(2 * groups * kTsluCols + 2 + kTsluCols) * sizeof(int) + size_t(2 * kTsluCols) * sizeof(int2) + 256;
}

cudaError_t tslu_identity(int32_t* perm, int64_t n, cudaStream_t s) {
  iota_kernel<<<cdivu(n, 256), 256, 0, s>>>(perm, n);
  return launched();
}

cudaError_t tslu_panel(void* Ap, int64_t m, int jb, int64_t lda, void* scratch, int64_t n_max, int* d_status,
                       cudaStream_t s) {
  if (jb <= 0 || jb > kTsluCols || m < jb || m > n_max) return cudaErrorInvalidValue;
  ProfScope prof("lu_panel", s, 4.0 * double(m) * jb * jb);
  float2* A = static_cast<float2*>(Ap);
  const int64_t groups_max = std::max<int64_t>((n_max + 2047) / 2048, 16);
  int2* moves = static_cast<int2*>(scratch);
  int* idx[2] = {reinterpret_cast<int*>(moves + 2 * kTsluCols), nullptr};
  idx[1] = idx[0] + groups_max * kTsluCols;
  int* last = idx[1] + groups_max * kTsluCols;  // [2]
  int* sel = last + 2;
  if (max_clusters(128) < 1 || max_clusters(256) < 1) return cudaErrorInvalidConfiguration;
  // A group has 64 places for nominees and the next level reads them all, but a panel narrower than
  // that fills only jb of them: its rows have to fit one level (the last panel of a matrix has m = jb).
  if (jb < kTsluCols && plan_level(m).clusters > 1) return cudaErrorInvalidValue;
  uint64_t nl = 0;
  int64_t rows = m;
  int groups = 0, cur = 0;
  for (;;) {
    const Level lv = plan_level(rows);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(lv.clusters * lv.cl));
    cfg.blockDim = dim3(kTsluThreads);
    cfg.dynamicSmemBytes = lv.rows_per_cta == 256 ? sizeof(PanelSmem<256>) : sizeof(PanelSmem<128>);
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = unsigned(lv.cl);
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    // leaves: an even share of at least 64 rows each, so that only the last group can be short;
    // merges: whole groups
    const int64_t rows_per = (rows + lv.clusters - 1) / lv.clusters;
    const int fan = lv.cl * lv.rows_per_cta / kTsluCols;
    const int* in = nl ? idx[cur] : nullptr;
    const int* in_last = last + cur;
    const int out = nl ? cur ^ 1 : 0;
    auto launch = [&](auto kern) {
      return cudaLaunchKernelEx(&cfg, kern, A, lda, m, jb, rows_per, in, groups, fan, in_last, idx[out], last + out,
                                sel, moves, d_status);
    };
    const cudaError_t e = lv.cl == 1 ? (lv.rows_per_cta == 256 ? launch(panel_cluster_kernel<256, 1>)
                                                               : launch(panel_cluster_kernel<128, 1>))
                                     : (lv.rows_per_cta == 256 ? launch(panel_cluster_kernel<256, kTsluCluster>)
                                                               : launch(panel_cluster_kernel<128, kTsluCluster>));
    if (e != cudaSuccess) return e;
    ++nl;
    if (lv.clusters == 1) break;
    cur = out;
    groups = lv.clusters;
    rows = int64_t(groups) * kTsluCols;
  }
  if (m > jb) {
    static bool ls_attr[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (!ls_attr[dev]) {
      const cudaError_t e = cudaFuncSetAttribute(tslu_lsolve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 int(kLsSmem));
      if (e != cudaSuccess) return e;
      ls_attr[dev] = true;
    }
    tslu_lsolve_kernel<<<cdivu(m - jb, kTriVec), kTriThreads, kLsSmem, s>>>(A, lda, m, jb);
    ++nl;
  }
  return launched(nl);
}

cudaError_t tri_lower_unit_cols(const void* D, int64_t ldd, int jb, void* X, int64_t ldx, int64_t ncols,
                                cudaStream_t s) {
  if (jb <= 0 || jb > kTsluCols) return cudaErrorInvalidValue;
  if (ncols <= 0) return cudaSuccess;
  tri_lower_unit_cols_kernel<<<cdivu(ncols, kTriVec), kTriThreads, 0, s>>>(static_cast<const float2*>(D), ldd, jb,
                                                                         static_cast<float2*>(X), ldx, ncols);
  return launched();
}

cudaError_t tslu_swap(void* A, int64_t n, int64_t lda, int64_t j0, int jb, const void* scratch, int32_t* perm,
                      cudaStream_t s) {
  if (jb <= 0 || jb > kTsluCols) return cudaErrorInvalidValue;
  tslu_swap_kernel<<<cdivu(n, 32), 256, 0, s>>>(static_cast<float2*>(A), n, lda, j0, jb,
                                                static_cast<const int2*>(scratch), perm);
  return launched();
}

}  // namespace fosb
