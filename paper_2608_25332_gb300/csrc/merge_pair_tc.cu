// Sec. 4.3, last paragraph: every pruned visual token joins its cosine-nearest
// kept token. The pruned x kept Gram fused with the row argmax, on pairs of SMs
// (tcgen05 cta_group::2).
//
// The operands are rows of E_v, fetched where they lie (direct), or contiguous rows
// of a per-sample copy of E_v permuted to [pruned | kept] (gather_perm_kernel): the
// copy reads and writes all of E_v, the direct form loads slower (see
// merge_pair_search). A unit of work is a tile (sample b,
// 512-row group q of its pruned positions, range t of its kept positions):
// the group's rows as two M = 256 halves (A0 = the first 256, A1 = the next
// 256) against the range's kept rows c0 .. c0+N-1 (N <= 256). The two CTAs of
// a cluster issue, from the even CTA, one M = 256 MMA per half and K step;
// CTA r (0 or 1) holds rows 128r .. 128r+127 of each half and kept rows
// c0 + r*N/2 .. c0 + r*N/2 + N/2 - 1 of B, and receives rows 128r .. 128r+127
// of both accumulators in its own tensor memory (columns 0 .. N-1 for A0,
// 256 .. 256+N-1 for A1). Each SM thus loads 48 KiB (its A rows and half of
// B) per 64-element K slice of a 256-column tile, against 64 KiB when one SM
// runs both M = 128 halves against all of B, and its MMAs read its half of B
// once for both SMs.
//
// A group splits its kept columns into n_lo or n_lo + 1 ranges (see
// pair_tile); the tiles are dealt to the clusters in snake order (see
// pair_deal_tile), so that the busiest pair of SMs gets as little work as the
// ranges allow, and the tiles of one group run side by side on different pairs
// and share its A rows through L2. Each CTA loads only the N/2 kept rows its
// half of the MMA reads (of the copy: one tensor map per distinct N/2 of the plan).
//
// Where 512-row groups are too few for the pairs of SMs (a few hundred pruned rows
// per sample), groups of 256 rows, one M = 256 half each, make twice the tiles
// (kHalves = 1): a K slice is then at most 32 KiB per SM, and six stages fit.
// merge_pair_best takes the form whose busiest pair has the fewest clocks.
//
// The epilogue (eight warps: two per TMEM lane quadrant, each taking half of
// the 32-column pieces, their tensor-memory loads double-buffered) scales
// column k by 1/|e_k| and keeps per row the running (max, first index) over
// its columns in ascending kept position; range t of a row writes slot t of
// the partials, which merge_assign_kernel combines (ties to the lower kept
// position).
//
// Every wait is bounded; a CTA that times out marks itself failed, and both
// CTAs drain to the closing cluster barrier, after which each frees its half
// of the pair's tensor memory. Before that barrier each producer waits for the
// MMAs' releases of its last stages and the MMA issuer for both epilogues'
// release of the last tile, so that no arrival lands in a CTA that has exited.
#include "common.cuh"
#include "kernels.h"
#include "merge_epi.cuh"
#include "tc_gemm.cuh"

#include <math.h>

#include <algorithm>
#include <mutex>
#include <vector>

namespace provip {
namespace {

using namespace tcg;

constexpr int kPairMaxN = 256;                     // columns of a tile
// by the M = 256 halves of a group (1 or 2): ring depth, bytes of a stage (A0 rows
// | A1 rows | B rows of this CTA), one accumulator per half
__host__ __device__ constexpr int pair_stages(int halves) { return halves == 2 ? 4 : 6; }
__host__ __device__ constexpr int pair_stage_bytes(int halves) { return (halves + 1) * kABytes; }
__host__ __device__ constexpr uint32_t pair_tmem_cols(int halves) { return (uint32_t)halves * kPairMaxN; }
constexpr int kPairEpiWarps = 8;                   // two per TMEM lane quadrant, splitting the columns
// warps that load: warp 0, and with rows fetched where they lie those past the
// epilogue's
__host__ __device__ constexpr int pair_load_warps(bool direct) { return direct ? 11 : 1; }
__host__ __device__ constexpr int pair_threads(bool direct) {
  return 32 * (1 + kPairEpiWarps + pair_load_warps(direct));
}

struct PairArgs {
  const int* pruned;    // [B][n_pruned] original row of each pruned position
  int n_pruned;
  const int* keep_idx;  // [B][keep]
  int keep;
  int N_v, D, B;
  const float* inv_v;   // [B][N_v]
  MergePairPlan plan;   // tiles and their deal to the pairs
  float* ws_best;       // [plan.n_slots][B][N_v]
  int* ws_bidx;
  unsigned* err;
};

// tensor maps of the permuted copy: A boxes of 128 rows, B boxes of each
// distinct half-width of the plan's tiles (so that a CTA loads only the N/2
// kept rows its half of the MMA reads); direct: a, of E_v, its boxes one row high
struct PairMaps {
  CUtensorMap a;
  CUtensorMap b[kMergePairHeights];
};

template <int kStages>
struct PairPipe {
  uint64_t full[kStages];   // even CTA: both CTAs' boxes of the stage have landed
  uint64_t empty[kStages];  // each CTA: the MMAs that read its stage are done
  uint64_t acc_full;            // each CTA: the tile's accumulators are complete
  uint64_t acc_empty;           // even CTA: both CTAs' epilogues have read them
  uint32_t tmem;
  volatile int fail;
};

__device__ __forceinline__ uint32_t pair_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of `local`'s counterpart in cluster CTA `rank`
__device__ __forceinline__ uint32_t cluster_addr(const void* local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(local)), "r"(rank));
  return r;
}
__device__ __forceinline__ void pair_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// tensor memory of the CTA pair: one warp of each CTA takes part
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* smem_result, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(smem_result)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
// D (+)= A * B^T over the CTA pair: M = 256 (128 rows of A and N/2 rows of B
// from each CTA's shared memory at the same offsets), bf16 in, fp32 out.
__device__ __forceinline__ void mma_pair_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                              uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrive on the mbarrier at `bar`'s offset in both CTAs of the pair once every
// MMA issued so far by this thread has completed
__device__ __forceinline__ void commit_pair(uint64_t* bar) {
  const uint16_t both = 0x3;
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 "
      "[%0], %1;" ::"r"(smem_u32(bar)),
      "h"(both)
      : "memory");
}
// 2-D tiled load into this CTA's shared memory whose completion is counted on
// an mbarrier of either CTA of the pair (bar: shared::cluster address)
__device__ __forceinline__ void tma_load_2d_pair(void* smem_dst, const CUtensorMap* map, int x, int y,
                                                 uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
// rows y0 .. y3 of 64 columns from x, 128 bytes each, one after the other
__device__ __forceinline__ void tma_gather4_pair(void* smem_dst, const CUtensorMap* map, int x, int y0, int y1, int y2,
                                                 int y3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y0), "r"(y1), "r"(y2), "r"(y3), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait on a barrier that the other CTA of the pair also signals
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, unsigned* err) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const unsigned long long t0 = global_timer_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((it & 63u) == 0 && global_timer_ns() - t0 > kWaitBudgetNs) {
      set_error(err, kErrTimeout);
      return false;
    }
  }
}

// every epilogue thread passes its predicate; all get the AND (a barrier of
// the epilogue warps)
__device__ __forceinline__ bool epilogue_all(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred q, p;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, 1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"(v ? 1u : 0u), "n"(32 * kPairEpiWarps)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ void epilogue_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(32 * kPairEpiWarps) : "memory");
}
// Tile k of the plan. Quads are numbered b * n_quads + q; quads x_hi .. Q-1
// split their kept columns into n_lo ranges and come first (tiles 0 ..
// (Q - x_hi) * n_lo - 1, the wider ones), quads 0 .. x_hi-1 into n_lo + 1.
// Range t of n starts at t * keep / n rounded down to a multiple of 32.
struct PairTile {
  int b, m0, t, n, c0, nv, N;
  bool has1;
};
__host__ __device__ __forceinline__ int pair_range_start(int t, int n, int keep) {
  return t == 0 ? 0 : (t >= n ? keep : (int)((long long)t * keep / n) & ~31);
}
__host__ __device__ __forceinline__ PairTile pair_tile(const MergePairPlan& p, int n_pruned, int keep, int k) {
  PairTile g;
  const int n_wide = (p.Q - p.x_hi) * p.n_lo;
  int quad;
  if (k < n_wide) {
    g.n = p.n_lo;
    quad = p.x_hi + k / p.n_lo;
    g.t = k % p.n_lo;
  } else {
    g.n = p.n_lo + 1;
    quad = (k - n_wide) / g.n;
    g.t = (k - n_wide) % g.n;
  }
  g.b = quad / p.n_quads;
  g.m0 = (quad % p.n_quads) * p.halves * 2 * kBM;
  g.has1 = p.halves == 2 && g.m0 + 2 * kBM < n_pruned;  // the second half holds pruned rows
  g.c0 = pair_range_start(g.t, g.n, keep);
  g.nv = pair_range_start(g.t + 1, g.n, keep) - g.c0;
  g.N = (g.nv + 31) / 32 * 32;         // MMA width: N / 2 rows of B per CTA, a multiple of 16
  return g;
}
// Tile of pair p in deal r (snake order: pairs 0 .. P-1 take tiles r*P ..
// in deals 0, 2, ..., and in reverse order in deals 1, 3, ..., so that a
// pair given one of the first, wider tiles gets one of the last, narrower ones);
// -1 past the last tile.
__host__ __device__ __forceinline__ int pair_deal_tile(const MergePairPlan& p, int pair, int r) {
  const int k = (r & 1) ? (r + 1) * p.P - 1 - pair : r * p.P + pair;
  return k < p.T ? k : -1;
}

template <int kHalves, bool kDirect>
__global__ void __launch_bounds__(pair_threads(kDirect), 1)
    merge_argmax_pair_tc(const PairArgs a, const __grid_constant__ PairMaps maps) {
  constexpr int kPairStages = pair_stages(kHalves), kPairStageBytes = pair_stage_bytes(kHalves);
  constexpr uint32_t kPairTmemCols = pair_tmem_cols(kHalves);
  constexpr uint32_t kBOff = kHalves * kABytes;  // B rows in a stage
  extern __shared__ uint8_t smem_raw[];
  __shared__ PairPipe<kPairStages> pipe;
  __shared__ int sidx[2 * kBM];      // original rows of this CTA's A0 and A1 rows (-1: none)
  __shared__ float skinv[kPairMaxN];  // 1/|e_k| of the tile's kept columns
  __shared__ float xbest[2][kBM];     // the upper column half's (max, position) per row
  __shared__ int xidx[2][kBM];
  const uint32_t rank = pair_rank();  // 0: issues the MMAs; 1: its peer
  const int pair = (int)(blockIdx.x >> 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_k = (a.D + kBK - 1) / kBK;
  const MergePairPlan& pl = a.plan;

  const uint32_t sbase = smem_u32(smem_raw);
  uint8_t* stages = smem_raw + (((sbase + 1023u) & ~1023u) - sbase);

  if (threadIdx.x == 0) {
    prefetch_tmap(&maps.a);
    for (int j = 0; !kDirect && j < pl.n_heights; ++j) prefetch_tmap(&maps.b[j]);
    for (int s = 0; s < kPairStages; ++s) {
      mbar_init(&pipe.full[s], 1);
      mbar_init(&pipe.empty[s], 1);
    }
    mbar_init(&pipe.acc_full, 1);
    mbar_init(&pipe.acc_empty, 2 * kPairEpiWarps);  // one arrival per epilogue warp of each CTA
    pipe.fail = 0;
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc_pair(&pipe.tmem, kPairTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  pair_cluster_sync();  // both CTAs' barriers initialised, the pair's tensor memory allocated
  tc_fence_after();
  // launched as a programmatic dependent of the kernel before: the set-up above ran
  // under its tail; the rows' copy and the index tables are read after this
  pdl_wait_prior();
  pdl_allow_next();

  // the MMAs' releases of the last stages land in this CTA before it may exit
  auto drain = [&](int it) {
    for (int i = it; i < it + kPairStages && !pipe.fail; ++i)
      if (!mbar_wait(&pipe.empty[i % kPairStages], ((uint32_t)(i / kPairStages) & 1u) ^ 1u, a.err)) pipe.fail = 1;
  };
  // loader warps: 0, then those past the epilogue's (2 .. 1 + kPairEpiWarps)
  const int loader = warp == 0 ? 0 : (warp >= 2 + kPairEpiWarps ? warp - 1 - kPairEpiWarps : -1);
  if (kDirect && loader >= 0) {
    // Both CTAs load their rows of every stage, four to a load: 32 loads for the 128
    // rows of each half, then N / 8 for the B rows, dealt to the loaders' lanes (one
    // each); completion counts on the even CTA's full barrier, which expects the bytes
    // of both. Positions past the last pruned or kept row repeat it (computed, never
    // stored).
    constexpr int kLoaders = pair_load_warps(true), kLoads = 32 * (kHalves + 1);
    constexpr int kPer = (kLoads + kLoaders - 1) / kLoaders;
    static_assert(kPer <= 32, "a load per lane");
    const int unit = loader * kPer + lane, area = unit / 32;
    const bool used = lane < kPer && unit < kLoads, bs = area == kHalves;
    auto rows_of = [&](int k, int* y) {
      const PairTile g = pair_tile(pl, a.n_pruned, a.keep, k);
      const int* list = bs ? a.keep_idx + (size_t)g.b * a.keep : a.pruned + (size_t)g.b * a.n_pruned;
      const int last = (bs ? a.keep : a.n_pruned) - 1;
      const int p0 = (bs ? g.c0 + (int)rank * (g.N / 2) : g.m0 + area * 2 * kBM + (int)rank * kBM) + 4 * (unit % 32);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        int j = list[min(p0 + e, last)];
        if (j < 0 || j >= a.N_v) {
          set_error(a.err, kErrBadDeviceArg);
          j = 0;
        }
        y[e] = g.b * a.N_v + j;
      }
    };
    const uint32_t full0 = cluster_addr(&pipe.full[0], 0);
    int it = 0;
    bool ok = true;
    int next[4] = {0, 0, 0, 0};
    int k = pair_deal_tile(pl, pair, 0);
    if (k >= 0 && used) rows_of(k, next);
    for (int rd = 1; k >= 0 && ok; ++rd) {
      const PairTile g = pair_tile(pl, a.n_pruned, a.keep, k);
      const int y0 = next[0], y1 = next[1], y2 = next[2], y3 = next[3];
      k = pair_deal_tile(pl, pair, rd);
      if (k >= 0 && used) rows_of(k, next);  // the next tile's rows, under this one's loads
      const bool mine = used && (bs ? unit % 32 < g.N / 8 : (area == 0 || g.has1));
      const uint32_t tx = 2u * (uint32_t)((g.has1 ? 2 : 1) * kABytes + (g.N / 2) * kBK * 2);
      for (int kb = 0; kb < n_k; ++kb, ++it) {
        const int s = it % kPairStages;
        const uint32_t ph = (uint32_t)(it / kPairStages) & 1u;
        if (lane == 0) ok = !pipe.fail && mbar_wait(&pipe.empty[s], ph ^ 1u, a.err);
        __syncwarp();  // orders the other lanes' loads after lane 0's wait; the shuffle alone does not
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        if (!ok) {
          pipe.fail = 1;
          break;
        }
        if (loader == 0 && rank == 0 && lane == 0) mbar_arrive_expect_tx(&pipe.full[s], tx);
        if (mine)
          tma_gather4_pair(stages + (size_t)s * kPairStageBytes + unit * (4 * kBK * 2), &maps.a, kb * kBK, y0, y1, y2,
                           y3, full0 + 8u * (uint32_t)s);
      }
    }
    if (loader == 0 && lane == 0) drain(it);
  } else if (!kDirect && warp == 0) {
    if (lane == 0) {
      // both CTAs load their rows of every stage; completion counts on the
      // even CTA's full barrier, which expects the bytes of both
      int it = 0;
      for (int rd = 0, k; (k = pair_deal_tile(pl, pair, rd)) >= 0 && !pipe.fail; ++rd) {
        const PairTile g = pair_tile(pl, a.n_pruned, a.keep, k);
        const int row_a = g.b * a.N_v + g.m0 + (int)rank * kBM;
        const int row_b = g.b * a.N_v + a.n_pruned + g.c0 + (int)rank * (g.N / 2);
        int hj = 0, hrows = pl.heights[0];  // the B map whose box height is N / 2
#pragma unroll
        for (int j = 1; j < kMergePairHeights; ++j)
          if (j < pl.n_heights && pl.heights[j] == g.N / 2) {
            hj = j;
            hrows = pl.heights[j];
          }
        const CUtensorMap* mapB = maps.b + hj;
        const uint32_t tx = 2u * (uint32_t)((g.has1 ? 2 : 1) * kABytes + hrows * kBK * 2);
        for (int kb = 0; kb < n_k; ++kb, ++it) {
          const int s = it % kPairStages;
          const uint32_t ph = (uint32_t)(it / kPairStages) & 1u;
          if (pipe.fail || !mbar_wait(&pipe.empty[s], ph ^ 1u, a.err)) {
            pipe.fail = 1;
            break;
          }
          uint8_t* sa = stages + (size_t)s * kPairStageBytes;
          const uint32_t fb = cluster_addr(&pipe.full[s], 0);
          const int x = kb * kBK;
          if (rank == 0) mbar_arrive_expect_tx(&pipe.full[s], tx);
          tma_load_2d_pair(sa, &maps.a, x, row_a, fb);
          if (kHalves == 2 && g.has1) tma_load_2d_pair(sa + kABytes, &maps.a, x, row_a + 2 * kBM, fb);
          tma_load_2d_pair(sa + kBOff, mapB, x, row_b, fb);
        }
      }
      drain(it);
    }
  } else if (warp == 1) {
    if (rank == 0 && lane == 0) {
      int it = 0, ti = 0;
      for (int rd = 0, k; (k = pair_deal_tile(pl, pair, rd)) >= 0; ++rd, ++ti) {
        const PairTile g = pair_tile(pl, a.n_pruned, a.keep, k);
        // both epilogues have read the previous tile's accumulators
        if (!pipe.fail && !mbar_wait_cluster(&pipe.acc_empty, ((uint32_t)ti & 1u) ^ 1u, a.err)) pipe.fail = 1;
        tc_fence_after();
        const uint32_t idesc = idesc_bf16_f32(2 * kBM, g.N);
        for (int kb = 0; kb < n_k; ++kb, ++it) {
          const int s = it % kPairStages;
          const uint32_t ph = (uint32_t)(it / kPairStages) & 1u;
          if (pipe.fail || !mbar_wait_cluster(&pipe.full[s], ph, a.err)) {
            pipe.fail = 1;
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(stages + (size_t)s * kPairStageBytes);
          const uint32_t sb = sa + kBOff;
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k) {
            const uint32_t acc = (kb > 0 || k > 0) ? 1u : 0u;
            const uint64_t bd = smem_desc_sw128(sb + k * 32);
            mma_pair_bf16(pipe.tmem, smem_desc_sw128(sa + k * 32), bd, idesc, acc);
            if (kHalves == 2 && g.has1) mma_pair_bf16(pipe.tmem + kPairMaxN, smem_desc_sw128(sa + kABytes + k * 32), bd, idesc, acc);
          }
          commit_pair(&pipe.empty[s]);  // frees stage s in both CTAs
        }
        commit_pair(&pipe.acc_full);  // arrives in both CTAs when every MMA above has completed
        if (pipe.fail) break;
      }
      // both epilogues' releases of the last tile land before this CTA may exit
      if (!pipe.fail && !mbar_wait_cluster(&pipe.acc_empty, ((uint32_t)ti & 1u) ^ 1u, a.err)) pipe.fail = 1;
    }
  } else {
    // epilogue: thread = TMEM lane = row of this CTA's half of A0 and of A1;
    // the two warps of a lane quadrant take the lower and the upper half of
    // the tile's 32-column chunks, and the lower merges the upper's result
    const int et = threadIdx.x - 64;
    const int quad = warp & 3;
    const int half = (warp - 2) / 4;
    const int r = quad * 32 + lane;
    const uint32_t acc_empty = cluster_addr(&pipe.acc_empty, 0);
    int ti = 0;
    for (int rd = 0, k; (k = pair_deal_tile(pl, pair, rd)) >= 0; ++rd, ++ti) {
      const PairTile g = pair_tile(pl, a.n_pruned, a.keep, k);
      const int* pr = a.pruned + (size_t)g.b * a.n_pruned;
      const int* kp = a.keep_idx + (size_t)g.b * a.keep;
      for (int i = et; i < kHalves * kBM; i += 32 * kPairEpiWarps) {
        const int pos = g.m0 + (i < kBM ? 0 : 2 * kBM) + (int)rank * kBM + (i & (kBM - 1));
        sidx[i] = pos < a.n_pruned ? pr[pos] : -1;
      }
      for (int q = et; q < g.nv; q += 32 * kPairEpiWarps) {
        int j = kp[g.c0 + q];
        if (j < 0 || j >= a.N_v) {
          set_error(a.err, kErrBadDeviceArg);
          j = 0;
        }
        skinv[q] = a.inv_v[(size_t)g.b * a.N_v + j];
      }
      RowBest r0, r1;
      r0.init();
      r1.init();
      // the epilogue warps agree on the outcome, so that they leave the loop
      // together (the barrier also completes the tables)
      const bool ok = epilogue_all(warp_mbar_wait(&pipe.acc_full, (uint32_t)ti & 1u, a.err) && !pipe.fail);
      if (ok) {
        tc_fence_after();
        const uint32_t taddr = pipe.tmem + ((uint32_t)(quad * 32) << 16);
        const int ncb = g.N / 32, mid = (ncb + 1) / 2;
        const int cb0 = half ? mid : 0, cb1 = half ? ncb : mid;
        // 32-column pieces (chunk cb of A0, then of A1 when the group has a
        // second half), double-buffered: piece j + 1 loads while j is reduced
        const int sh = kHalves == 2 && g.has1 ? 1 : 0;
        const int npc = (cb1 - cb0) << sh;
        auto piece = [&](int j, float* v) {
          tmem_ld32(taddr + (uint32_t)((j & sh) * kPairMaxN + (cb0 + (j >> sh)) * 32), v);
        };
        auto reduce = [&](int j, const float* v) {
          const int cb = cb0 + (j >> sh);
          if (j & sh)
            r1.add32(v, skinv + cb * 32, cb * 32, g.nv, g.c0);
          else
            r0.add32(v, skinv + cb * 32, cb * 32, g.nv, g.c0);
        };
        float va[32], vb[32];
        if (npc > 0) piece(0, va);
#pragma unroll 1
        for (int j = 0; j < npc; j += 2) {
          tc_wait_ld_into(va);
          if (j + 1 < npc) piece(j + 1, vb);
          reduce(j, va);
          if (j + 1 < npc) {
            tc_wait_ld_into(vb);
            if (j + 2 < npc) piece(j + 2, va);
            reduce(j + 1, vb);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acc_empty);  // this warp is done with the accumulators
      if (!ok) {
        pipe.fail = 1;
        break;
      }
      float best0, best1;
      int bidx0, bidx1;
      r0.result(best0, bidx0);
      r1.result(best1, bidx1);
      if (half) {
        xbest[0][r] = best0;
        xidx[0][r] = bidx0;
        xbest[1][r] = best1;
        xidx[1][r] = bidx1;
      }
      epilogue_sync();  // the upper halves' results are in shared memory
      if (!half) {
        // the upper half's positions are all larger: it wins only if larger
        if (xbest[0][r] > best0) {
          best0 = xbest[0][r];
          bidx0 = xidx[0][r];
        }
        if (xbest[1][r] > best1) {
          best1 = xbest[1][r];
          bidx1 = xidx[1][r];
        }
        const size_t slot = (size_t)a.B * a.N_v;
        const size_t o = ((size_t)g.t * a.B + g.b) * a.N_v;
        // the last range of a quad with fewer ranges than slots also fills the
        // spare slot with an entry that never wins
        const bool spare = g.t + 1 == g.n && g.n < pl.n_slots;
        const int j0 = sidx[r];
        if (j0 >= 0) {
          a.ws_best[o + j0] = best0;
          a.ws_bidx[o + j0] = bidx0;
          if (spare) {
            a.ws_best[o + slot + j0] = -INFINITY;
            a.ws_bidx[o + slot + j0] = 0x7fffffff;
          }
        }
        if constexpr (kHalves == 2) {
          const int j1 = sidx[kBM + r];
          if (g.has1 && j1 >= 0) {
            a.ws_best[o + j1] = best1;
            a.ws_bidx[o + j1] = bidx1;
            if (spare) {
              a.ws_best[o + slot + j1] = -INFINITY;
              a.ws_bidx[o + slot + j1] = 0x7fffffff;
            }
          }
        }
      }
      epilogue_sync();  // tables and exchange free for the next tile
    }
  }
  tc_fence_before();
  __syncwarp();
  pair_cluster_sync();  // every MMA of the pair has completed and been read
  if (warp == 0) tmem_dealloc_pair(pipe.tmem, kPairTmemCols);
}

size_t pair_smem(int halves) { return (size_t)pair_stages(halves) * pair_stage_bytes(halves) + 1024; }

// per device: 0 = not checked, 1 = two-CTA clusters of both forms fit, 2 = they do not
std::atomic<int> g_pair_ok[64];
std::atomic<int> g_pair_enabled{1};

}  // namespace

void merge_pair_enable(int on) { g_pair_enabled.store(on ? 1 : 0); }

// Tiles and their deal for B samples of n_pruned pruned and keep kept rows
// of width D on num_sms SMs: among splits that give 1 to 4 tiles per pair of
// SMs (and the even splits), the one whose busiest pair has the fewest clocks
// by a model of a tile of N columns: per 64-element K slice the larger of its
// MMA clocks (4N with both halves of the group, 2N with one) and the ring's pace,
// plus 9000 clocks of epilogue and refill per tile, plus the copy's clocks where the
// rows are not read where they lie. The pace of boxes of the copy: a stage's loads
// take about 2700 clocks from issue to landing, 960 with four stages of 48 KiB in
// shared memory; 760 to 800 measured with six of at most 32. Rows fetched four to a
// load come slower (paces of 900 to 1100 and of 1300 to 1500 measured): it takes a
// warp some 150 clocks to issue a load, so that many warps share them, and the SM
// begins one every 14 clocks at best. The pass of 32 images (576 rows of width 5120)
// took 196, 181, 178, 172 and 174 us with 4, 6, 8, 11 and 12 of them; on the copy,
// which alone takes 52 (378 MB), 219. 8 of 2880 rows of width 4096: 256 -> 216; 16
// images of width 4096: 231 -> 221; 4 of 1443 rows: 135 -> 132. A video of 9216 rows
// of width 3584 keeps the copy (179 us against 182). Slower than either: 16-byte
// cp.async by eight warps (243 us for the 32 images: too few requests fit in flight
// beside the ring), and copying the kept rows alone (191 us).
constexpr long long kBoxPace[2] = {780, 960};         // by halves
constexpr long long kDirectPace[2] = {1090, 1400};
constexpr double kCopyClocksPerByte = 1.9 / 7200;     // 7.2 TB/s, read and write, at 1.9 GHz
// plan[0]: the best split for boxes of the copy, plan[1]: for rows read where they lie
// (ok: found). Both forms share each candidate's deal, which is walked tile by tile, and
// only where the mean load of its pairs is below the best busiest pair so far.
static void merge_pair_search(int halves, int B, int n_pruned, int keep, int D, int num_sms, MergePairPlan* plan,
                              bool* ok) {
  ok[0] = ok[1] = false;
  if (B < 1 || n_pruned < 1 || keep < 1 || D < 1 || num_sms < 2) return;
  const int quad_rows = halves * 2 * kBM;
  const int n_quads = (n_pruned + quad_rows - 1) / quad_rows;
  const long long pace[2] = {kBoxPace[halves - 1], kDirectPace[halves - 1]};
  const double copy[2] = {kCopyClocksPerByte * 4.0 * B * (n_pruned + keep) * (double)D, 0.0};
  const long long Q = (long long)B * n_quads;
  const int max_pairs = num_sms / 2;
  const long long n_k = (D + kBK - 1) / kBK;
  if (Q > (1 << 20)) return;
  // whether the last group of a sample, or every group, holds one half
  const bool last_one = halves == 1 || n_pruned - (n_quads - 1) * quad_rows <= 2 * kBM, all_one = halves == 1;
  long long best[2] = {0, 0};
  std::vector<long long> load[2];
  auto consider = [&](int n_lo, long long x_hi) {
    const int n_hi = n_lo + (x_hi > 0 ? 1 : 0);
    if (n_lo < 1 || n_hi > kMergeMaxSplit || x_hi < 0 || x_hi >= Q) return;
    MergePairPlan c;
    c.halves = halves;
    c.n_quads = n_quads;
    c.Q = (int)Q;
    c.n_lo = n_lo;
    c.x_hi = (int)x_hi;
    const long long T = x_hi * (n_lo + 1) + (Q - x_hi) * n_lo;
    if (T > (1 << 24)) return;
    c.T = (int)T;
    c.P = (int)(T < max_pairs ? T : max_pairs);
    c.n_slots = n_hi;
    c.n_heights = 0;
    // clocks of a range's tile by form, number of ranges (n_lo, n_hi) and halves of its
    // group, and of a group's tiles together
    long long cost[2][2][2][kMergeMaxSplit], row[2][2][2] = {};
    for (int n = n_lo; n <= n_hi; ++n)
      for (int t = 0; t < n; ++t) {
        const int nv = pair_range_start(t + 1, n, keep) - pair_range_start(t, n, keep);
        if (nv < 1 || nv > kPairMaxN) return;
        const int N = (nv + 31) / 32 * 32, h = N / 2;  // B rows per CTA
        int j = 0;
        while (j < c.n_heights && c.heights[j] != h) ++j;
        if (j == c.n_heights) {
          if (j == kMergePairHeights) return;
          c.heights[c.n_heights++] = h;
        }
        for (int f = 0; f < 2; ++f)
          for (int two = 0; two < 2; ++two) {
            const long long v = n_k * std::max((two ? 4ll : 2ll) * N, pace[f]) + 9000;
            cost[f][n - n_lo][two][t] = v;
            row[f][n - n_lo][two] += v;
          }
      }
    // groups of one half among the first x_hi and among the others
    const long long one_hi = all_one ? x_hi : (last_one ? x_hi / n_quads : 0);
    const long long one_lo = (all_one ? Q : (last_one ? B : 0)) - one_hi;
    bool try_form[2];
    for (int f = 0; f < 2; ++f) {
      const int hi = n_hi - n_lo;
      const long long total = one_hi * row[f][hi][0] + (x_hi - one_hi) * row[f][hi][1] + one_lo * row[f][0][0] +
                              (Q - x_hi - one_lo) * row[f][0][1];
      try_form[f] = !ok[f] || total < best[f] * c.P;  // else its busiest pair has at least best[f]
    }
    if (!try_form[0] && !try_form[1]) return;
    // the tiles in order (pair_tile), dealt in snake order (pair_deal_tile)
    for (int f = 0; f < 2; ++f) load[f].assign((size_t)c.P, 0);
    int pr = 0, step = 1;
    for (int part = 0; part < 2; ++part) {
      const long long q0 = part == 0 ? x_hi : 0, q1 = part == 0 ? Q : x_hi;
      int in_sample = (int)(q0 % n_quads);
      for (long long q = q0; q < q1; ++q) {
        const int two = !(all_one || (last_one && in_sample == n_quads - 1));
        if (++in_sample == n_quads) in_sample = 0;
        const long long *c0 = cost[0][part][two], *c1 = cost[1][part][two];
        for (int t = 0; t < n_lo + part; ++t) {
          load[0][pr] += c0[t];
          load[1][pr] += c1[t];
          pr += step;
          if (pr == c.P || pr < 0) {
            step = -step;
            pr += step;
          }
        }
      }
    }
    for (int f = 0; f < 2; ++f) {
      if (!try_form[f]) continue;
      const long long worst = *std::max_element(load[f].begin(), load[f].end());
      if (!ok[f] || worst < best[f]) {
        ok[f] = true;
        best[f] = worst;
        plan[f] = c;
        plan[f].direct = f == 1;
        plan[f].clocks = (double)worst + copy[f];
      }
    }
  };
  for (int n_lo = (keep + kPairMaxN - 1) / kPairMaxN; n_lo <= kMergeMaxSplit; ++n_lo) {
    consider(n_lo, 0);
    for (int m = 1; m <= 4; ++m) {
      const long long x_hi = (long long)m * max_pairs - Q * n_lo;
      if (x_hi > 0 && x_hi < Q) consider(n_lo, x_hi);
    }
  }
}

// The searches take 3 to 7 us of host time for the shapes above and 7 for 64 x 2880 rows
// (four searches that dealt every candidate took 120, 400 and 2600): their results are
// kept per shape, the last kPlanCache shapes, for the calls that follow.
namespace {
constexpr int kPlanCache = 16;
struct PlanEntry {
  int B, n_pruned, keep, D, num_sms;
  bool ok[2];             // by halves - 1
  MergePairPlan plan[2];
};
std::mutex g_plan_mu;
PlanEntry g_plans[kPlanCache];
int g_plan_n = 0, g_plan_next = 0;
}  // namespace

// both group sizes' plans, each in the form with the fewer clocks
static PlanEntry plans_of(int B, int n_pruned, int keep, int D, int num_sms) {
  {
    std::lock_guard<std::mutex> lock(g_plan_mu);
    for (int i = 0; i < g_plan_n; ++i) {
      const PlanEntry& e = g_plans[i];
      if (e.B == B && e.n_pruned == n_pruned && e.keep == keep && e.D == D && e.num_sms == num_sms) return e;
    }
  }
  PlanEntry e{B, n_pruned, keep, D, num_sms, {}, {}};
  for (int h = 0; h < 2; ++h) {
    MergePairPlan form[2];
    bool ok[2];
    merge_pair_search(h + 1, B, n_pruned, keep, D, num_sms, form, ok);
    e.ok[h] = ok[0] || ok[1];
    if (e.ok[h]) e.plan[h] = ok[1] && (!ok[0] || form[1].clocks < form[0].clocks) ? form[1] : form[0];
  }
  std::lock_guard<std::mutex> lock(g_plan_mu);
  g_plans[g_plan_next] = e;
  g_plan_next = (g_plan_next + 1) % kPlanCache;
  if (g_plan_n < kPlanCache) ++g_plan_n;
  return e;
}

static bool plan_of(int halves, int B, int n_pruned, int keep, int D, int num_sms, MergePairPlan* p) {
  const PlanEntry e = plans_of(B, n_pruned, keep, D, num_sms);
  if (e.ok[halves - 1]) *p = e.plan[halves - 1];
  return e.ok[halves - 1];
}
bool merge_pair_plan(int B, int n_pruned, int keep, int D, int num_sms, MergePairPlan* p) {
  return plan_of(2, B, n_pruned, keep, D, num_sms, p);
}
bool merge_pair_half_plan(int B, int n_pruned, int keep, int D, int num_sms, MergePairPlan* p) {
  return plan_of(1, B, n_pruned, keep, D, num_sms, p);
}

// Measured: 16 samples of 288 pruned by 288 kept rows, 64 tiles of 256 rows on the 76
// pairs instead of 32 of 512: 41 -> 31 us (of the copy); 4 of 962 by 481: 41 -> 30;
// 32 of 384 by 192 (width 5120): 50 -> 44. 8 of 1920 by 960 keep 512-row groups (84 us): 256-row
// tiles would take four rounds of the pairs instead of two.
bool merge_pair_best(int B, int n_pruned, int keep, int D, int num_sms, MergePairPlan* p) {
  const PlanEntry e = plans_of(B, n_pruned, keep, D, num_sms);
  if (e.ok[0] && (!e.ok[1] || e.plan[0].clocks < e.plan[1].clocks)) {
    *p = e.plan[0];
  } else if (e.ok[1]) {
    *p = e.plan[1];
  }
  return e.ok[0] || e.ok[1];
}

bool merge_pair_usable(const SimArgs& a) {
  if (!g_pair_enabled.load() || a.dtype != 1 || a.D % 8) return false;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  int st = g_pair_ok[dev].load(std::memory_order_acquire);
  if (st == 0) {
    st = 2;
    auto fits = [](auto kernel, int halves, bool direct) {
      const size_t smem = pair_smem(halves);
      cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 2;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.gridDim = dim3(2, 1, 1);
      cfg.blockDim = dim3(pair_threads(direct), 1, 1);
      cfg.dynamicSmemBytes = smem;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int n = 0;
      e = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg);
      return e == cudaSuccess && n < 1 ? cudaErrorInvalidConfiguration : e;
    };
    cudaError_t e = fits(merge_argmax_pair_tc<2, false>, 2, false);
    if (e == cudaSuccess) e = fits(merge_argmax_pair_tc<1, false>, 1, false);
    if (e == cudaSuccess) e = fits(merge_argmax_pair_tc<2, true>, 2, true);
    if (e == cudaSuccess) e = fits(merge_argmax_pair_tc<1, true>, 1, true);
    if (e == cudaSuccess) st = 1;
    // a refused attribute or query falls back to the single-SM form: clear the
    // error it left (only then, so that no earlier error of the caller is lost)
    if (e != cudaSuccess) cudaGetLastError();
    g_pair_ok[dev].store(st, std::memory_order_release);
  }
  return st == 1;
}

cudaError_t merge_argmax_pair_launch(const SimArgs& a, const int* keep_idx, int keep, const float* inv_v,
                                     const int* pruned, const void* perm, const MergePairPlan& plan,
                                     float* ws_best, int* ws_bidx, cudaStream_t s) {
  PairMaps maps;
  const uint64_t rows = (uint64_t)a.B * a.N_v;
  if (make_tmap_bf16_2d(&maps.a, plan.direct ? a.emb_v : perm, rows, (uint64_t)a.D, (uint64_t)a.D * 2,
                        plan.direct ? 1 : kBM))
    return cudaErrorInvalidValue;
  for (int j = 0; !plan.direct && j < plan.n_heights; ++j)
    if (make_tmap_bf16_2d(&maps.b[j], perm, rows, (uint64_t)a.D, (uint64_t)a.D * 2, (uint32_t)plan.heights[j]))
      return cudaErrorInvalidValue;
  PairArgs m;
  m.pruned = pruned;
  m.n_pruned = a.N_v - keep;
  m.keep_idx = keep_idx;
  m.keep = keep;
  m.N_v = a.N_v;
  m.D = a.D;
  m.B = a.B;
  m.inv_v = inv_v;
  m.plan = plan;
  m.ws_best = ws_best;
  m.ws_bidx = ws_bidx;
  m.err = a.err;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3((unsigned)(2 * plan.P), 1, 1);
  cfg.blockDim = dim3(pair_threads(plan.direct), 1, 1);
  cfg.dynamicSmemBytes = pair_smem(plan.halves);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  auto go = [&](auto kernel) { return cudaLaunchKernelEx(&cfg, kernel, m, maps); };
  if (plan.direct) return plan.halves == 2 ? go(merge_argmax_pair_tc<2, true>) : go(merge_argmax_pair_tc<1, true>);
  return plan.halves == 2 ? go(merge_argmax_pair_tc<2, false>) : go(merge_argmax_pair_tc<1, false>);
}

}  // namespace provip
