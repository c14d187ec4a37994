// Pre-LLM pass (Sec. 4.3) on 5th-generation tensor cores (bf16).
//
// merge_argmax_tc: the pruned x kept cosine Gram fused with the row argmax, on
//   single SMs (the form on pairs of SMs is merge_pair_tc.cu, the default).
//   A = the pruned visual rows of two 128-row M tiles, B = the kept rows of a
//   range of 256-row N tiles shared by both, read as contiguous tiles of a
//   per-sample copy of E_v permuted to [pruned | kept] by one bandwidth-bound
//   gather pass. The epilogue scales a column by 1/|e_k| and keeps, per row,
//   the running (max, first index) over the kept positions in ascending order,
//   so ties go to the lower kept position. The (N_v - N1) x N1 matrix never
//   leaves the SM.
// relevance_fused_tc: the visual x [visual ; text] Gram of a 128-row visual
//   tile, one read of the visual rows giving |v_j|^2 (the diagonal of the
//   visual block), the cosines and the de-meaning sums (p_j itself is formed by
//   a small second kernel once every tile's sums are known).
// crit_gram_tc: the text Gram E_t E_t^T, split over K in a cluster, and up to 128
//   text rows the whole of Sec. 4.2 in the same kernel.
#include "common.cuh"
#include "kernels.h"
#include "merge_epi.cuh"
#include "tc_gemm.cuh"

namespace provip {
namespace {

using namespace tcg;

// perm[b] = rows of E_v[b] reordered as [pruned rows (ascending) | kept rows
// (keep order)], so that the Gram reads both operands as contiguous tiles.
// One warp per output row, 16-byte vectors.
__global__ void __launch_bounds__(256) gather_perm_kernel(const __nv_bfloat16* E, const int* pruned,
                                                          const int* keep_idx, int n_pruned, int keep,
                                                          int N_v, int D, __nv_bfloat16* perm,
                                                          unsigned* err) {
  pdl_wait_prior();  // pruned and keep_idx come from the kernels before
  pdl_allow_next();  // the Gram may set itself up meanwhile
  const int b = blockIdx.y;
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= N_v) return;
  int j = r < n_pruned ? pruned[(size_t)b * n_pruned + r] : keep_idx[(size_t)b * keep + (r - n_pruned)];
  if (j < 0 || j >= N_v) {
    if (lane == 0) set_error(err, kErrBadDeviceArg);
    j = 0;
  }
  const uint4* src = reinterpret_cast<const uint4*>(E + ((size_t)b * N_v + j) * D);
  uint4* dst = reinterpret_cast<uint4*>(perm + ((size_t)b * N_v + r) * D);
  const int nvec = D / 8;
  // four 16-byte loads in flight per lane before their stores
  int v = lane;
  for (; v + 96 < nvec; v += 128) {
    const uint4 x0 = __ldg(src + v), x1 = __ldg(src + v + 32), x2 = __ldg(src + v + 64), x3 = __ldg(src + v + 96);
    dst[v] = x0;
    dst[v + 32] = x1;
    dst[v + 64] = x2;
    dst[v + 96] = x3;
  }
  for (; v < nvec; v += 32) dst[v] = __ldg(src + v);
}

struct MergeTcArgs {
  const int* pruned;   // [B][n_pruned]
  int n_pruned;
  const int* keep_idx; // [B][keep]
  int keep;
  int N_v, D, B;
  const float* inv_v;  // [B][N_v]
  int n_split;
  float* ws_best;      // [n_split][B][N_v]
  int* ws_bidx;
  unsigned* err;
};

constexpr int kMergeBN = 256;
constexpr int kMergeMaxKeep = 2560;  // kept rows handled by one split (shared index table)
constexpr int kMergeStages = 3;
constexpr int kMergeBBytes = kMergeBN * kBK * 2;                 // 32 KiB
constexpr int kMergeStageBytes = 2 * kABytes + kMergeBBytes;     // A0 | A1 | B: 64 KiB
constexpr uint32_t kMergeTmemCols = 2 * kMergeBN;                // one accumulator per M tile
constexpr int kMergeEpiWarps = 8;  // two per TMEM lane quadrant, splitting each tile's columns
constexpr int kMergeThreads = 64 + 32 * kMergeEpiWarps;

struct MergePipe {
  uint64_t full[kMergeStages];
  uint64_t empty[kMergeStages];
  uint64_t acc_full;
  uint64_t acc_empty;
  uint32_t tmem;
  volatile int fail;
};

// One CTA owns two 128-row M tiles of pruned rows (A0, A1) and sweeps its range
// of 256-row N tiles of kept rows; each stage holds A0, A1 and one B tile, and
// two MMAs (M = 128, N <= 256) share that B tile, so a stage carries 64 KiB for
// 8.4 MFLOP instead of 48 KiB for 4.2 MFLOP with a single M tile. The two
// accumulators fill the 512 TMEM columns: the epilogue of an N tile runs
// between that tile's last MMA and the next tile's first (the producer keeps
// loading meanwhile), so it is kept short: eight warps, two per TMEM lane
// quadrant, each taking half of a tile's 32-column pieces with its loads
// double-buffered and four interleaved running maxima per row (RowBest). The
// last N tile's MMA is only as wide as its kept rows (rounded up to 16).
__global__ void __launch_bounds__(kMergeThreads, 1)
    merge_argmax_tc(const MergeTcArgs a, const __grid_constant__ CUtensorMap mapE) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ MergePipe pipe;
  __shared__ int sidx_a[2 * kBM];
  __shared__ float xbest[2][kBM];  // the upper column halves' (max, position) per row
  __shared__ int xidx[2][kBM];
  const int b = blockIdx.z, split = blockIdx.y;
  const int m0 = blockIdx.x * 2 * kBM;
  const bool has1 = m0 + kBM < a.n_pruned;  // the second M tile holds pruned rows
  const int n_tiles_all = (a.keep + kMergeBN - 1) / kMergeBN;
  const int t0 = (int)((long long)n_tiles_all * split / a.n_split);
  const int t1 = (int)((long long)n_tiles_all * (split + 1) / a.n_split);
  const int n_tiles = t1 - t0;
  const int a0 = t0 * kMergeBN;                       // first kept position of the range
  const int n_keep = min(a.keep, t1 * kMergeBN) - a0;  // kept rows in the range
  const int n_k = (a.D + kBK - 1) / kBK;

  const uint32_t sbase = smem_u32(smem_raw);
  uint8_t* stages = smem_raw + (((sbase + 1023u) & ~1023u) - sbase);
  float* skinv = reinterpret_cast<float*>(stages + (size_t)kMergeStages * kMergeStageBytes);

  if (threadIdx.x == 0) {
    prefetch_tmap(&mapE);
    for (int s = 0; s < kMergeStages; ++s) {
      mbar_init(&pipe.full[s], 1);
      mbar_init(&pipe.empty[s], 1);
    }
    mbar_init(&pipe.acc_full, 1);
    mbar_init(&pipe.acc_empty, kMergeEpiWarps);  // one arrival per epilogue warp
    pipe.fail = 0;
    fence_mbar_init();
  }
  if (threadIdx.x < 32) {
    tmem_alloc(&pipe.tmem, kMergeTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  // N columns of tile t: 256, or the kept rows of a ragged last tile rounded up to 16
  auto tile_cols = [&](int t) { return min(kMergeBN, (n_keep - t * kMergeBN + 15) / 16 * 16); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (n_tiles > 0) {
    if (warp == 0) {
      if (lane == 0) {
        // operands are contiguous rows of the permuted copy [pruned | kept];
        // rows past a tile's valid rows are computed and never used
        const int row_a = b * a.N_v + m0;
        const int row_b = b * a.N_v + a.n_pruned + a0;
        int it = 0;
        for (int t = 0; t < n_tiles && !pipe.fail; ++t) {
          const bool b_hi = tile_cols(t) > kBM;  // the tile's second 128-row box is used
          const uint32_t tx = (uint32_t)((has1 ? 2 : 1) * kABytes + (b_hi ? 2 : 1) * kABytes);
          for (int kb = 0; kb < n_k; ++kb, ++it) {
            const int s = it % kMergeStages;
            const uint32_t ph = (uint32_t)(it / kMergeStages) & 1u;
            if (pipe.fail || !mbar_wait(&pipe.empty[s], ph ^ 1u, a.err)) {
              pipe.fail = 1;
              break;
            }
            uint8_t* sa = stages + (size_t)s * kMergeStageBytes;
            uint8_t* sb = sa + 2 * kABytes;
            const int x = kb * kBK;
            mbar_arrive_expect_tx(&pipe.full[s], tx);
            tma_load_2d(sa, &mapE, x, row_a, &pipe.full[s]);
            if (has1) tma_load_2d(sa + kABytes, &mapE, x, row_a + kBM, &pipe.full[s]);
            tma_load_2d(sb, &mapE, x, row_b + t * kMergeBN, &pipe.full[s]);
            if (b_hi) tma_load_2d(sb + kABytes, &mapE, x, row_b + t * kMergeBN + kBM, &pipe.full[s]);
          }
        }
      }
    } else if (warp == 1) {
      if (lane == 0) {
        int it = 0;
        for (int t = 0; t < n_tiles; ++t) {
          if (!pipe.fail && !mbar_wait(&pipe.acc_empty, ((uint32_t)t & 1u) ^ 1u, a.err)) pipe.fail = 1;
          const uint32_t idesc = idesc_bf16_f32(kBM, tile_cols(t));
          for (int kb = 0; kb < n_k; ++kb, ++it) {
            const int s = it % kMergeStages;
            const uint32_t ph = (uint32_t)(it / kMergeStages) & 1u;
            if (pipe.fail || !mbar_wait(&pipe.full[s], ph, a.err)) {
              pipe.fail = 1;
              break;
            }
            tc_fence_after();
            const uint32_t sa = smem_u32(stages + (size_t)s * kMergeStageBytes);
            const uint32_t sb = sa + 2 * kABytes;
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k) {
              const uint32_t acc = (kb > 0 || k > 0) ? 1u : 0u;
              const uint64_t bd = smem_desc_sw128(sb + k * 32);
              tc_mma_bf16(pipe.tmem, smem_desc_sw128(sa + k * 32), bd, idesc, acc);
              if (has1) tc_mma_bf16(pipe.tmem + kMergeBN, smem_desc_sw128(sa + kABytes + k * 32), bd, idesc, acc);
            }
            tc_commit(&pipe.empty[s]);
          }
          tc_commit(&pipe.acc_full);  // arrives when every MMA above has completed
          if (pipe.fail) break;
        }
      }
    } else {
      // the epilogue warps fill the index tables while the first stages load
      const int* pr = a.pruned + (size_t)b * a.n_pruned;
      const int* kp = a.keep_idx + (size_t)b * a.keep;
      const int et = threadIdx.x - 64;
      constexpr int kEpi = 32 * kMergeEpiWarps;
      for (int r = et; r < 2 * kBM; r += kEpi) sidx_a[r] = m0 + r < a.n_pruned ? pr[m0 + r] : 0;
      for (int q = et; q < n_keep; q += kEpi) {
        int j = kp[a0 + q];
        if (j < 0 || j >= a.N_v) {
          set_error(a.err, kErrBadDeviceArg);
          j = 0;
        }
        skinv[q] = a.inv_v[(size_t)b * a.N_v + j];
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kEpi) : "memory");  // tables complete (epilogue warps)
      // epilogue: row r of each M tile; the two warps of a lane quadrant take
      // the lower and the upper half of each tile's 32-column pieces (their
      // tensor-memory loads double-buffered), each keeping a running (max,
      // first position) over the range, merged at the end
      const int quad = warp & 3;
      const int half = (warp - 2) / 4;
      const int r = quad * 32 + lane;
      RowBest r0, r1;
      r0.init();
      r1.init();
      bool ok = true;
      for (int t = 0; t < n_tiles; ++t) {
        ok = warp_mbar_wait(&pipe.acc_full, (uint32_t)t & 1u, a.err) && !pipe.fail;
        if (!ok) break;
        tc_fence_after();
        const uint32_t taddr = pipe.tmem + ((uint32_t)(quad * 32) << 16);
        const int ncb = (tile_cols(t) + 31) / 32, mid = (ncb + 1) / 2;
        const int cb0 = half ? mid : 0, cb1 = half ? ncb : mid;
        const int sh = has1 ? 1 : 0;
        const int npc = (cb1 - cb0) << sh;
        auto piece = [&](int j, float* v) {
          tmem_ld32(taddr + (uint32_t)((j & sh) * kMergeBN + (cb0 + (j >> sh)) * 32), v);
        };
        auto reduce = [&](int j, const float* v) {
          const int q0 = t * kMergeBN + (cb0 + (j >> sh)) * 32;  // position within the range
          if (j & sh)
            r1.add32(v, skinv + q0, q0, n_keep, a0);
          else
            r0.add32(v, skinv + q0, q0, n_keep, a0);
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
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&pipe.acc_empty);
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
      asm volatile("bar.sync 1, %0;" ::"n"(kEpi) : "memory");  // the upper halves' results
      if (!half) {
        if (merge_better(xbest[0][r], xidx[0][r], best0, bidx0)) {
          best0 = xbest[0][r];
          bidx0 = xidx[0][r];
        }
        if (merge_better(xbest[1][r], xidx[1][r], best1, bidx1)) {
          best1 = xbest[1][r];
          bidx1 = xidx[1][r];
        }
      }
      if (!half && ok && !pipe.fail) {
        const size_t o = ((size_t)split * a.B + b) * a.N_v;
        if (m0 + r < a.n_pruned) {
          a.ws_best[o + sidx_a[r]] = best0;
          a.ws_bidx[o + sidx_a[r]] = bidx0;
        }
        if (m0 + kBM + r < a.n_pruned) {
          a.ws_best[o + sidx_a[kBM + r]] = best1;
          a.ws_bidx[o + sidx_a[kBM + r]] = bidx1;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) tmem_dealloc(pipe.tmem, kMergeTmemCols);
}

// relevance_fused_tc: one read of the visual rows gives, per tile of R visual
// rows of sample b (R = 128, 96 or 64, chosen so that the tiles spread evenly
// over the SMs; A = the tile's rows, B = [the same R visual rows ; the text
// rows], both already adjacent in the stage, so one MMA of N = R + NT; the
// MMA's 128 A rows run past the R visual rows and their results are unused),
//   * |v_j|^2 from the diagonal of the visual x visual block (thread = TMEM
//     lane = visual row j reads its own column),
//   * the cosines Y[b][j][i] = <v_j, t_i> |t_i|^-1 |v_j|^-1 (|t_i|^-1 from a
//     separate pass over the text rows),
//   * the tile's column sums part[b][tile][i] = sum_j Y[b][j][i] (warp
//     butterfly, then the four lane quadrants in order).
// relevance_finish_kernel then forms mu_i = (sum of the tile sums in tile
// order) / N_v and p_j = max_{i in T} (Y[b][j][i] - mu_i) (Sec. 4.3).
// More than 128 text rows (kLong) are split into blocks of at most 128 (grid z); each
// block's CTAs read the visual tiles again (from L2, where the first block's
// loads left them), one CTA per SM with a deep ring. FFMA kernels took such texts
// before, 990 us for 4 x 1443 visual rows under 300 text rows, and their sums were rounded
// to nearest where the tensor core truncates at every accumulation: two accumulators
// over half of the K slices each left p further off than FFMA from width 3584 on
// (relative error against 64 bits on random rows 8.7e-7 at 4096 and 1.7e-6 at 8192, FFMA
// 6.0e-7 and 1.0e-6), and 1/|v_j|, which the merge reads on its own, 2.6e-6 and 5.2e-6 (FFMA
// 0.9e-7 and 1.3e-7). So here
//   * an accumulator takes kRelChunk slices, two in turn, and the epilogue warps add them up
//     in registers: p is 1.1e-7 off at widths 512 to 5120 and 2.5e-7 at 8192;
//   * warps of their own add up the squares of the visual rows from the slices as they
//     pass, each text block those of its share of the rows: 1/|v_j| is 0.4e-7 off at every
//     width.
// Both cost the K loop some 4%: the pass of the batch above 128.3 -> 130.3 us, 8 x 2880 rows
// 333 -> 337, 32 x 576 rows of width 5120 under 512 531 -> 540. With the squares of every row
// in the first block, whose CTAs then set the pace of a single wave: 132.8, 341 and 540; in
// its epilogue warps 349 for the 8 x 2880; by all blocks in place of the visual block of the
// MMA 355. Chunks of two and of eight slices: 360 and 342.
struct RelFusedArgs {
  int B, N_v, D, N_t_max;
  int NT;        // text rows in the MMA (a block's rows, a multiple of 16)
  int NTs;       // text columns of Y and part (N_t_max rounded up to 16)
  int R;         // visual rows per tile (128, 96 or 64)
  int n_vt;      // visual tiles per sample
  int n_stages;  // shared-memory ring depth
  const float* inv_t;  // [B][N_t_max]
  float* inv_v;  // [B][N_v]
  float* Y;      // [B][N_v][NTs]
  float* part;   // [B][n_vt][NTs]
  unsigned* err;
};

constexpr int kRelMaxStages = 8;
constexpr int kRelFinishRows = 8;  // rows per warp of relevance_finish_kernel
constexpr uint32_t kRelTmemCols = 256;  // 128 visual + <= 128 text columns

constexpr int kRelChunk = 4;            // K slices of an accumulator with several text blocks
constexpr int kRelSqWarps = 2;          // then more warps, for the squares of a block's share of the rows
constexpr int kRelLongThreads = kThreads + 32 * kRelSqWarps;

struct RelPipe {
  uint64_t full[kRelMaxStages];
  uint64_t empty[kRelMaxStages];
  uint64_t acc_full[2];   // one accumulator, or two in turn with several text blocks
  uint64_t acc_empty[2];
  uint32_t tmem;
  volatile int fail;
};

template <bool kLong>
__global__ void __launch_bounds__(kLong ? kRelLongThreads : kThreads, kLong ? 1 : 2)
    relevance_fused_tc(const RelFusedArgs a, const __grid_constant__ CUtensorMap mapV,
                       const __grid_constant__ CUtensorMap mapT) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ RelPipe pipe;
  __shared__ float s_invt[kBM];
  __shared__ float red[4][kBM];
  const int b = blockIdx.y, tile = blockIdx.x;
  const int tb0 = blockIdx.z * a.NT;  // first text row of the block
  const int R = a.R;
  const int n0 = tile * R;
  const int n_k = (a.D + kBK - 1) / kBK;
  const int NS = a.n_stages;
  const uint32_t st_bytes = (uint32_t)(R + a.NT) * 128u;
  constexpr uint32_t kCols = (kLong ? 2 : 1) * kRelTmemCols;
  const uint32_t sbase = smem_u32(smem_raw);
  uint8_t* stages = smem_raw + (((sbase + 1023u) & ~1023u) - sbase);
  if (threadIdx.x == 0) {
    prefetch_tmap(&mapV);
    prefetch_tmap(&mapT);
    for (int s = 0; s < NS; ++s) {
      mbar_init(&pipe.full[s], 1);
      mbar_init(&pipe.empty[s], kLong ? 1 + kRelSqWarps : 1);  // the MMAs, and the warps that add squares
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&pipe.acc_full[s], 1);
      mbar_init(&pipe.acc_empty[s], 4);  // the epilogue warps
    }
    pipe.fail = 0;
    fence_mbar_init();
  }
  if (threadIdx.x < 32) {
    tmem_alloc(&pipe.tmem, kCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) {
    if (lane == 0) {
      for (int kb = 0; kb < n_k; ++kb) {
        const int s = kb % NS;
        const uint32_t ph = (uint32_t)(kb / NS) & 1u;
        if (pipe.fail || !mbar_wait(&pipe.empty[s], ph ^ 1u, a.err)) {
          pipe.fail = 1;
          break;
        }
        uint8_t* sa = stages + (size_t)s * st_bytes;
        mbar_arrive_expect_tx(&pipe.full[s], st_bytes);
        // rows past the sample's last visual row belong to the next sample (or
        // lie past the tensor and read as zeros): computed, never stored
        tma_load_2d(sa, &mapV, kb * kBK, b * a.N_v + n0, &pipe.full[s]);
        tma_load_2d(sa + R * 128, &mapT, kb * kBK, b * a.N_t_max + tb0, &pipe.full[s]);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16_f32(kBM, R + a.NT);
      // One lane issues every MMA, and at some 800 clocks a slice it, not the loads, set the
      // pace: so it adds byte offsets, in 16-byte units, to the first stage's descriptor,
      // counts stages instead of dividing, and looks at the next slice's barriers before it
      // issues this one's MMAs.
      const uint64_t desc0 = smem_desc_sw128(smem_u32(stages));
      uint64_t desc = desc0;
      int s = 0, in_ch = 0;                // the slice's stage; its place in its accumulator
      uint32_t ph = 0, buf = 0, ph_a = 1;  // parities of full and, with several blocks, of acc_empty
      bool there = false, room = false;    // the next slice's loads and accumulator, looked at ahead
      for (int kb = 0; kb < n_k; ++kb) {
        if (kLong && in_ch == 0 && !room && !pipe.fail && !mbar_wait(&pipe.acc_empty[buf], ph_a, a.err)) pipe.fail = 1;
        if (pipe.fail || (!there && !mbar_wait(&pipe.full[s], ph, a.err))) {
          pipe.fail = 1;
          break;
        }
        const bool wrap = s + 1 == NS, last = kb == n_k - 1, ends = kLong && (in_ch + 1 == kRelChunk || last);
        const int s1 = wrap ? 0 : s + 1;
        const uint32_t ph1 = wrap ? ph ^ 1u : ph;
        there = !last && mbar_test(&pipe.full[s1], ph1);
        if (ends) room = !last && mbar_test(&pipe.acc_empty[buf ^ 1u], ph_a ^ buf);
        tc_fence_after();
        const uint32_t acc = pipe.tmem + buf * kRelTmemCols;
#pragma unroll
        for (int k = 0; k < kBK / 16; ++k)
          tc_mma_bf16(acc, desc + 2 * k, desc + 2 * k, idesc, ((kLong ? in_ch : kb) > 0 || k > 0) ? 1u : 0u);
        tc_commit(&pipe.empty[s]);
        desc = wrap ? desc0 : desc + (st_bytes >> 4);
        s = s1;
        ph = ph1;
        ++in_ch;
        if (ends) {
          tc_commit(&pipe.acc_full[buf]);  // arrives once every MMA above has completed
          in_ch = 0;
          ph_a ^= buf;  // the second accumulator's turn ends a round
          buf ^= 1u;
        }
      }
      if (!kLong) tc_commit(&pipe.acc_full[0]);
    }
  } else if (kLong && warp >= kThreads / 32) {
    static_assert(32 * kRelSqWarps >= kBM / 2, "a lane for each row of a block's share (two blocks or more)");
    // 1/|v_j| for the merge, of this block's share of the tile's rows, a lane each: the
    // squares of the row's slices as they pass, a slice's 64 in eight chains, the slices by
    // TwoSum (in one chain over the slices the sum is biased low: squares of bf16 values are
    // 0 or 1 mod 4 in their last place, so that rounding them to a longer one's goes down
    // more often). A row's eight 16-byte pieces lie in some order in its 128 bytes, and lane
    // l starts with piece l of them, so that eight lanes meet every bank.
    const int share = (R + (int)gridDim.z - 1) / (int)gridDim.z, q0 = (warp - kThreads / 32) * 32;
    const int r = (int)blockIdx.z * share + q0 + lane, j = n0 + r;
    const bool mine = q0 + lane < share && r < R;
    const uint8_t* row = stages + (size_t)(mine ? r : 0) * 128;
    float sum = 0.f, rest = 0.f;
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int kb = 0; kb < n_k && ok; ++kb) {
      ok = warp_mbar_wait(&pipe.full[s], ph, a.err);
      uint4 u[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        u[i] = *reinterpret_cast<const uint4*>(row + (size_t)s * st_bytes + ((i + lane) & 7) * 16);
      __syncwarp();
      if (lane == 0) mbar_arrive(&pipe.empty[s]);  // before the work on it
      if (++s == NS) {
        s = 0;
        ph ^= 1u;
      }
      float sq[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t w[4] = {u[i].x, u[i].y, u[i].z, u[i].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
          sq[2 * e] = fmaf(lo, lo, sq[2 * e]);
          sq[2 * e + 1] = fmaf(hi, hi, sq[2 * e + 1]);
        }
      }
      const float q = ((sq[0] + sq[1]) + (sq[2] + sq[3])) + ((sq[4] + sq[5]) + (sq[6] + sq[7]));
      const float t = sum + q, z = t - sum;
      rest += (sum - (t - z)) + (q - z);
      sum = t;
    }
    if (!ok) pipe.fail = 1;
    pdl_wait_prior();
    sum += rest;
    if (ok && mine && j < a.N_v) a.inv_v[(size_t)b * a.N_v + j] = sum > 0.f ? 1.f / sqrtf(sum) : 0.f;
  } else {
    const int quad = warp & 3;
    const int r = quad * 32 + lane;
    const int j = n0 + r;
    const bool rv = r < R && j < a.N_v;
    const uint32_t taddr = pipe.tmem + ((uint32_t)(quad * 32) << 16);
    const int nt = min(a.NT, a.NTs - tb0);  // the last block may be narrower
    float v[32];
    // |v_j|^2: column j of the visual block, i.e. element `lane` of the warp's 32 columns
    auto diagonal = [&]() {
      float d = 0.f;
#pragma unroll
      for (int i = 0; i < 32; ++i) d = i == lane ? v[i] : d;
      return d;
    };
    bool ok = true;
    float sqv = 0.f;
    float sum[kLong ? kBM : 1];  // several text blocks: the products, chunk by chunk
    if constexpr (kLong) {
#pragma unroll
      for (int i = 0; i < kBM; ++i) sum[i] = 0.f;
      const int n_ch = (n_k + kRelChunk - 1) / kRelChunk;
      for (int ch = 0; ch < n_ch && ok; ++ch) {
        ok = warp_mbar_wait(&pipe.acc_full[ch & 1], (uint32_t)(ch >> 1) & 1u, a.err);
        if (!ok) pipe.fail = 1;
        tc_fence_after();
        const uint32_t tch = taddr + ((ch & 1) ? kRelTmemCols : 0u);
        tmem_ld32(tch + (uint32_t)(quad * 32), v);
        tc_wait_ld_into(v);
        sqv += diagonal();
#pragma unroll
        for (int cb = 0; cb < kBM / 32; ++cb)
          if (cb * 32 < nt) {
            tmem_ld32(tch + (uint32_t)(R + cb * 32), v);
            tc_wait_ld_into(v);
#pragma unroll
            for (int i = 0; i < 32; ++i) sum[cb * 32 + i] += v[i];
          }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&pipe.acc_empty[ch & 1]);
      }
    }
    // launched as a programmatic dependent of the text-row norms: the loads and
    // MMAs ran under that kernel; its output (and every write below) waits here
    pdl_wait_prior();
    s_invt[r] = tb0 + r < a.N_t_max ? a.inv_t[(size_t)b * a.N_t_max + tb0 + r] : 0.f;
    asm volatile("bar.sync 1, 128;" ::: "memory");  // s_invt complete (epilogue warps)
    if constexpr (!kLong) {
      ok = warp_mbar_wait(&pipe.acc_full[0], 0, a.err);
      tc_fence_after();
    }
    ok = ok && !pipe.fail;
    pdl_allow_next();  // the finish kernel, where it follows without an event between
    if constexpr (!kLong) {
      tmem_ld32(taddr + (uint32_t)(quad * 32), v);
      tc_wait_ld();
      sqv = diagonal();
    }
    const float iv = sqv > 0.f ? 1.f / sqrtf(sqv) : 0.f;
    if (!kLong && rv && ok) a.inv_v[(size_t)b * a.N_v + j] = iv;
    float* yrow = a.Y + ((size_t)b * a.N_v + (rv ? j : 0)) * a.NTs + tb0;
    // the cosines of text columns [32 cb, ..), from the products in v, and their sums
    auto columns = [&](int cb) {
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = v[i] * s_invt[cb * 32 + i] * iv;
      if (rv && ok) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (cb * 32 + q * 4 < nt)
            *reinterpret_cast<float4*>(yrow + cb * 32 + q * 4) =
                make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      }
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = rv ? v[i] : 0.f;
      // butterfly sum over the 32 rows of the warp: lane ends with column `lane`
#pragma unroll
      for (int sh = 16; sh >= 1; sh >>= 1) {
        const bool upper = (lane & sh) != 0;
#pragma unroll
        for (int i = 0; i < sh; ++i) {
          const float keep = upper ? v[i + sh] : v[i];
          const float send = upper ? v[i] : v[i + sh];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, sh);
        }
      }
      red[quad][cb * 32 + lane] = v[0];
    };
    if constexpr (kLong) {
#pragma unroll
      for (int cb = 0; cb < kBM / 32; ++cb)
        if (cb * 32 < nt) {
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = sum[cb * 32 + i];
          columns(cb);
        }
    } else {
#pragma unroll 1
      for (int cb = 0; cb * 32 < nt; ++cb) {
        tmem_ld32(taddr + (uint32_t)(R + cb * 32), v);
        tc_wait_ld();
        columns(cb);
      }
    }
    tc_fence_before();
    asm volatile("bar.sync 1, 128;" ::: "memory");
    const int c = threadIdx.x - 64;
    if (c < nt && ok)
      a.part[((size_t)b * a.n_vt + tile) * a.NTs + tb0 + c] = (red[0][c] + red[1][c]) + (red[2][c] + red[3][c]);
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) tmem_dealloc(pipe.tmem, kCols);
}

// mu_i from the tile sums (tile order; every CTA forms all of mu), then p_j =
// max over the critical rows of Y[b][j][i] - mu_i; an empty T gives -inf.
__global__ void __launch_bounds__(256) relevance_finish_kernel(const RelFusedArgs a, const int* text_len,
                                                               const uint8_t* mask, float* p) {
  pdl_allow_next();  // the top-k reads p only after this grid completes
  pdl_wait_prior();  // the cosines, and the mask before them
  extern __shared__ float mu[];  // mu [NTs], valid [NTs]
  int* valid = reinterpret_cast<int*>(mu + a.NTs);
  const int b = blockIdx.y;
  const int tl = min(max(text_len[b], 0), a.N_t_max);
  for (int c = threadIdx.x; c < a.NTs; c += blockDim.x) {
    const bool v = c < tl && mask[(size_t)b * a.N_t_max + c] != 0;
    float s = 0.f;
    if (v) {
      const float* col = a.part + (size_t)b * a.n_vt * a.NTs + c;
      for (int t0 = 0; t0 < a.n_vt; t0 += 32) {
        float x[32];
#pragma unroll
        for (int u = 0; u < 32; ++u) x[u] = t0 + u < a.n_vt ? col[(size_t)(t0 + u) * a.NTs] : 0.f;
#pragma unroll
        for (int u = 0; u < 32; ++u)
          if (t0 + u < a.n_vt) s += x[u];
      }
    }
    mu[c] = s / (float)a.N_v;
    valid[c] = v;
  }
  __syncthreads();
  // a warp per kRelFinishRows rows: lane q reads the 16-byte pieces q, q + 32, ..
  // of each row (one piece up to 128 text rows), every row's load in flight, then
  // a warp max
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nq = a.NTs / 4;
  const int j0 = (blockIdx.x * (blockDim.x >> 5) + warp) * kRelFinishRows;
  const float4* y = reinterpret_cast<const float4*>(a.Y + (size_t)b * a.N_v * a.NTs);
  float best[kRelFinishRows];
#pragma unroll
  for (int r = 0; r < kRelFinishRows; ++r) best[r] = -INFINITY;
  for (int q = lane; q < nq; q += 32) {
    const int c = q * 4;
    const float m0 = mu[c], m1 = mu[c + 1], m2 = mu[c + 2], m3 = mu[c + 3];
    const bool v0 = valid[c], v1 = valid[c + 1], v2 = valid[c + 2], v3 = valid[c + 3];
    float4 f[kRelFinishRows];
#pragma unroll
    for (int r = 0; r < kRelFinishRows; ++r)
      f[r] = j0 + r < a.N_v ? y[(size_t)(j0 + r) * nq + q] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < kRelFinishRows; ++r) {
      if (v0) best[r] = fmaxf(best[r], f[r].x - m0);
      if (v1) best[r] = fmaxf(best[r], f[r].y - m1);
      if (v2) best[r] = fmaxf(best[r], f[r].z - m2);
      if (v3) best[r] = fmaxf(best[r], f[r].w - m3);
    }
  }
#pragma unroll
  for (int r = 0; r < kRelFinishRows; ++r) {
    const float m = warp_max(best[r]);
    if (lane == 0 && j0 + r < a.N_v) p[(size_t)b * a.N_v + j0 + r] = m;
  }
}

// The text Gram G = E_t E_t^T (Sec. 4.2): a cluster of C CTAs per 128 x 128 tile
// of a sample, each summing its share of the K slices in A of C x A accumulators
// (C x A = 16 parts: the sums are bound by the latency of a few small loads, so
// they are spread over CTAs, and short accumulation chains keep them exact to a
// few ulp). Each CTA adds its accumulators in order, puts the tile part in its
// shared memory and frees its tensor memory (before it waits for its peers, so
// that a CTA holding tensor memory never waits for one that wants it); then CTA
// c adds rows [c * 128 / C, ..) of the C parts in order over distributed shared
// memory.
// kWhole (at most 128 text rows: one tile): the rows are complete where they
// were added, so the same kernel goes on to their softmax (a warp per row), the
// column sums (rows of a warp, then warps, then CTAs, in order) and, in CTA 0,
// the mean and the mask. With the parts in global memory, added by a second
// kernel and finished by a third on one CTA per sample, the chain took
// 14 + 3 + 10 us for 8 samples of 96 rows and 29 + 5 + 14 for 16 of 128, longer
// than the relevance Gram it runs beside (the pre-LLM pass: 192 -> 185 us for a
// video, 275 -> 257 for the schedule of 16 images). Past 128 text rows the FFMA
// Gram took 330 us for 4 samples of 300 rows and the finish 34: the pass of
// that batch went from 605 to 148 us.
// Otherwise the rows go to G and crit_finish_kernel follows.
struct CritArgs {
  const int* text_len;
  int N_t_max, n_k;
  int nt;          // 128-row tiles per side
  int n_acc;       // accumulators per CTA
  float* G;        // [B][N_t_max][N_t_max]; unused with kWhole
  uint8_t* mask;   // kWhole: the outputs
  float* r_out;
  bool early;      // let the next kernel start beside this one
  unsigned* err;
};
constexpr int kCritStages = 4;
constexpr int kCritMaxAcc = 4;
constexpr int kCritLd = kBM + 4;  // padded row of the tile part in shared memory
constexpr int kCritMaxCluster = 8;

struct CritPipe {
  uint64_t full[kCritStages];
  uint64_t empty[kCritStages];
  uint64_t acc_full;
  uint32_t tmem;
  volatile int fail;
};

__device__ __forceinline__ void crit_cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(const void* local, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(local)), "r"(rank));
  return a;
}
__device__ __forceinline__ float4 ld_peer_f4(const float* local, uint32_t rank) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(peer_addr(local, rank))
               : "memory");
  return v;
}

template <bool kWhole>
__global__ void __launch_bounds__(kThreads, 1)
    crit_gram_tc(const CritArgs a, const __grid_constant__ CUtensorMap mapT) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ CritPipe pipe;
  __shared__ __align__(16) float wcol[kThreads / 32][kBM];
  __shared__ __align__(16) float ccol[kBM];
  __shared__ float wsum[4];
  __shared__ int wcnt[4];
  const uint32_t rank = blockIdx.x, C = gridDim.x;  // the cluster spans grid x
  const int ti = blockIdx.y / a.nt, tj = blockIdx.y % a.nt, b = blockIdx.z;
  const bool same = ti == tj;  // one load per K slice is both operands
  const int k0 = (int)((long long)a.n_k * rank / C), n = (int)((long long)a.n_k * (rank + 1) / C) - k0;
  const int n_acc = min(a.n_acc, n);  // n >= 1: C <= n_k
  const uint32_t sbase = smem_u32(smem_raw);
  uint8_t* stages = smem_raw + (((sbase + 1023u) & ~1023u) - sbase);
  constexpr uint32_t kStage = kWhole ? kABytes : 2 * kABytes;
  const uint32_t cols = (uint32_t)a.n_acc * kBM;
  if (threadIdx.x == 0) {
    prefetch_tmap(&mapT);
    for (int s = 0; s < kCritStages; ++s) {
      mbar_init(&pipe.full[s], 1);
      mbar_init(&pipe.empty[s], 1);
    }
    mbar_init(&pipe.acc_full, 1);
    pipe.fail = 0;
    fence_mbar_init();
  }
  if (threadIdx.x < 32) {
    tmem_alloc(&pipe.tmem, cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // Only now that this CTA has its tensor memory: the text norms that this lets start
  // let the relevance start, whose CTAs take tensor memory and keep it until the
  // norms, and through them this grid, have completed. A CTA of this grid that still
  // waited for its own could wait for ever. What waits for this grid does so in
  // inv_norm_kernel.
  if (a.early) pdl_allow_next();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* tile = reinterpret_cast<float*>(stages);  // [128][kCritLd], once the MMAs are done
  if (warp == 0) {
    if (lane == 0) {
      for (int i = 0; i < n; ++i) {
        const int s = i % kCritStages;
        if (pipe.fail || !mbar_wait(&pipe.empty[s], ((uint32_t)(i / kCritStages) & 1u) ^ 1u, a.err)) {
          pipe.fail = 1;
          break;
        }
        uint8_t* sa = stages + (size_t)s * kStage;
        mbar_arrive_expect_tx(&pipe.full[s], same ? kABytes : 2 * kABytes);
        tma_load_2d(sa, &mapT, (k0 + i) * kBK, b * a.N_t_max + ti * kBM, &pipe.full[s]);
        if (!same) tma_load_2d(sa + kABytes, &mapT, (k0 + i) * kBK, b * a.N_t_max + tj * kBM, &pipe.full[s]);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int q = -1;
      for (int i = 0; i < n; ++i) {
        const int s = i % kCritStages;
        if (pipe.fail || !mbar_wait(&pipe.full[s], (uint32_t)(i / kCritStages) & 1u, a.err)) {
          pipe.fail = 1;
          break;
        }
        tc_fence_after();
        const bool first = q != i * n_acc / n;  // the accumulator's first slice
        q = i * n_acc / n;
        const uint32_t sa = smem_u32(stages + (size_t)s * kStage);
        const uint32_t sb = same ? sa : sa + kABytes;
#pragma unroll
        for (int k = 0; k < kBK / 16; ++k)
          tc_mma_bf16(pipe.tmem + (uint32_t)q * kBM, smem_desc_sw128(sa + k * 32), smem_desc_sw128(sb + k * 32),
                      idesc_bf16_f32(kBM, kBM), (!first || k > 0) ? 1u : 0u);
        tc_commit(&pipe.empty[s]);
      }
      tc_commit(&pipe.acc_full);  // arrives once every MMA above has completed
    }
  } else {
    const int quad = warp & 3;
    const int r = quad * 32 + lane;
    warp_mbar_wait(&pipe.acc_full, 0, a.err);
    tc_fence_after();
    const uint32_t taddr = pipe.tmem + ((uint32_t)(quad * 32) << 16);
#pragma unroll 1
    for (int cb = 0; cb < kBM / 32; ++cb) {
      float v[32];
      tmem_ld32(taddr + cb * 32, v);
      tc_wait_ld_into(v);
#pragma unroll 1
      for (int q = 1; q < n_acc; ++q) {
        float w[32];
        tmem_ld32(taddr + (uint32_t)q * kBM + cb * 32, w);
        tc_wait_ld_into(w);
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] += w[i];
      }
#pragma unroll
      for (int i = 0; i < 32; i += 4)
        *reinterpret_cast<float4*>(tile + (size_t)r * kCritLd + cb * 32 + i) =
            make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) tmem_dealloc(pipe.tmem, cols);
  crit_cluster_sync();  // every part of the tile is in its CTA's shared memory

  const int n_rows = kBM / (int)C;  // rows that this CTA adds and owns
  // row i of its share, columns [4 lane, 4 lane + 4): the parts in order
  auto gram4 = [&](int i) {
    const float* src = tile + (size_t)((int)rank * n_rows + i) * kCritLd + lane * 4;
    float4 v[kCritMaxCluster];
#pragma unroll
    for (uint32_t q = 0; q < kCritMaxCluster; ++q)
      if (q < C) v[q] = ld_peer_f4(src, q);
    float4 g = v[0];
#pragma unroll
    for (uint32_t q = 1; q < kCritMaxCluster; ++q)
      if (q < C) {
        g.x += v[q].x;
        g.y += v[q].y;
        g.z += v[q].z;
        g.w += v[q].w;
      }
    return g;
  };
  if (!kWhole) {
    for (int i = warp; i < n_rows; i += kThreads / 32) {
      const float4 g = gram4(i);
      const int row = ti * kBM + (int)rank * n_rows + i, col = tj * kBM + lane * 4;
      if (row < a.N_t_max && !pipe.fail) {
        float* o = a.G + ((size_t)b * a.N_t_max + row) * a.N_t_max + col;
        const float ge[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (col + e < a.N_t_max) o[e] = ge[e];
      }
    }
    crit_cluster_sync();  // no CTA leaves while a peer may still read its part
    return;
  }
  int tl = a.text_len[b];
  if (tl < 0 || tl > a.N_t_max) {
    if (rank == 0 && threadIdx.x == 0) set_error(a.err, kErrBadDeviceArg);
    tl = 0;
  }
  float4 cs = make_float4(0.f, 0.f, 0.f, 0.f);
  const int c0 = lane * 4;
  for (int i = warp; i < n_rows; i += kThreads / 32) {
    if ((int)rank * n_rows + i >= tl) break;  // warp-uniform
    const float4 g = gram4(i);
    const float gv[4] = {c0 < tl ? g.x : -INFINITY, c0 + 1 < tl ? g.y : -INFINITY,
                         c0 + 2 < tl ? g.z : -INFINITY, c0 + 3 < tl ? g.w : -INFINITY};
    const float m = warp_max(fmaxf(fmaxf(gv[0], gv[1]), fmaxf(gv[2], gv[3])));
    float e[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) e[q] = c0 + q < tl ? expf(gv[q] - m) : 0.f;
    const float inv = 1.f / warp_sum((e[0] + e[1]) + (e[2] + e[3]));
    cs.x += e[0] * inv;
    cs.y += e[1] * inv;
    cs.z += e[2] * inv;
    cs.w += e[3] * inv;
  }
  *reinterpret_cast<float4*>(&wcol[warp][c0]) = cs;
  __syncthreads();
  const int j = threadIdx.x;
  if (j < kBM) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) s += wcol[w][j];
    ccol[j] = s;
  }
  crit_cluster_sync();  // every CTA's column sums
  float r = 0.f;
  if (rank == 0) {
    if (j < kBM) {
      for (uint32_t q = 0; q < C; ++q) {
        float v;
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(peer_addr(&ccol[j], q)) : "memory");
        r += v;
      }
      r = j < tl ? r / (float)tl : 0.f;
      const float s = warp_sum(r);
      if (lane == 0) wsum[warp] = s;
    }
    __syncthreads();
    const float mean = tl > 0 ? ((wsum[0] + wsum[1]) + (wsum[2] + wsum[3])) / (float)tl : 0.f;
    const bool over = j < tl && r > mean;
    if (j < kBM) {
      const unsigned bal = __ballot_sync(0xffffffffu, over);
      if (lane == 0) wcnt[warp] = __popc(bal);
    }
    __syncthreads();
    const int cnt = (wcnt[0] + wcnt[1]) + (wcnt[2] + wcnt[3]);
    if (j < a.N_t_max) {
      a.mask[(size_t)b * a.N_t_max + j] = (j < tl && (cnt == 0 || over)) ? 1 : 0;
      if (a.r_out) a.r_out[(size_t)b * a.N_t_max + j] = r;
    }
  }
  crit_cluster_sync();  // no CTA leaves while CTA 0 may still read its column sums
}

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes, std::atomic<bool>* done) {
  if (done->load()) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) done->store(true);  // idempotent: concurrent first calls may both set it
  return e;
}

}  // namespace

size_t merge_tc_smem() {
  return (size_t)kMergeStages * kMergeStageBytes + 1024 + (size_t)kMergeMaxKeep * sizeof(float);
}

int merge_tc_split(int B, int N_v, int keep, int num_sms) {
  const int m_tiles = B * ((N_v - keep + 2 * kBM - 1) / (2 * kBM));  // CTAs: pairs of M tiles
  const int n_tiles = (keep + kMergeBN - 1) / kMergeBN;
  int best = 1;
  long long best_cost = -1;
  for (int sp = 1; sp <= n_tiles && sp <= kMergeMaxSplit; ++sp) {
    const int per = (n_tiles + sp - 1) / sp;
    if (per * kMergeBN > kMergeMaxKeep) continue;
    const long long waves = ((long long)m_tiles * sp + num_sms - 1) / num_sms;
    const long long cost = waves * per;
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best = sp;
    }
  }
  return best;
}

bool merge_tc_supported(const SimArgs& a, int keep, int n_split) {
  if (a.dtype != 1 || a.D % 8) return false;
  const int n_tiles = (keep + kMergeBN - 1) / kMergeBN;
  const int per_split = (n_tiles + n_split - 1) / n_split;
  return per_split * kMergeBN <= kMergeMaxKeep && keep < a.N_v;
}

cudaError_t merge_argmax_tc_launch(const SimArgs& a, const int* keep_idx, int keep, const float* inv_v,
                                   const int* pruned, void* perm, int n_split,
                                   float* ws_best, int* ws_bidx, int num_sms, int* n_split_out,
                                   cudaStream_t s) {
  const int n_pruned = a.N_v - keep;  // pruned: the rows not kept, ascending (merge_index_kernel)
  MergePairPlan plan;
  const bool pairs = merge_pair_usable(a) && merge_pair_best(a.B, n_pruned, keep, a.D, num_sms, &plan);
  cudaError_t e = cudaSuccess;
  if (!pairs) {
    static std::atomic<bool> smem_set[64];  // per device, zero-initialised
    int dev = 0;
    cudaGetDevice(&dev);
    e = set_smem(merge_argmax_tc, merge_tc_smem(), &smem_set[dev < 64 ? dev : 0]);
    if (e != cudaSuccess) return e;
  }
  dim3 gg((a.N_v + 7) / 8, a.B);
  if (!pairs || !plan.direct)
    e = launch_pdl(gather_perm_kernel, gg, dim3(256), 0, s, static_cast<const __nv_bfloat16*>(a.emb_v), pruned,
                   keep_idx, n_pruned, keep, a.N_v, a.D, static_cast<__nv_bfloat16*>(perm), a.err);
  if (e != cudaSuccess) return e;
  if (pairs) {
    *n_split_out = plan.n_slots;
    return merge_argmax_pair_launch(a, keep_idx, keep, inv_v, pruned, perm, plan, ws_best, ws_bidx, s);
  }
  *n_split_out = n_split;
  const size_t smem = merge_tc_smem();
  CUtensorMap mapE;
  if (make_tmap_bf16_2d(&mapE, perm, (uint64_t)a.B * a.N_v, (uint64_t)a.D, (uint64_t)a.D * 2, 128))
    return cudaErrorInvalidValue;
  MergeTcArgs m;
  m.pruned = pruned;
  m.n_pruned = n_pruned;
  m.keep_idx = keep_idx;
  m.keep = keep;
  m.N_v = a.N_v;
  m.D = a.D;
  m.B = a.B;
  m.inv_v = inv_v;
  m.n_split = n_split;
  m.ws_best = ws_best;
  m.ws_bidx = ws_bidx;
  m.err = a.err;
  dim3 grid((n_pruned + 2 * kBM - 1) / (2 * kBM), n_split, a.B);
  merge_argmax_tc<<<grid, kMergeThreads, smem, s>>>(m, mapE);
  return cudaGetLastError();
}

// up to the text rows that the finish kernel's shared memory holds (32 KiB)
constexpr int kRelMaxNt = 4096;
bool relevance_tc_supported(const SimArgs& a) { return a.dtype == 1 && a.N_t_max <= kRelMaxNt && a.D % 8 == 0; }

static int rel_nt(int N_t_max) { return (N_t_max + 15) / 16 * 16; }

size_t relevance_fused_floats(int B, int N_v, int N_t_max) {
  const int NT = rel_nt(N_t_max), n_vt = (N_v + 63) / 64;  // tiles of the smallest R
  return (size_t)B * N_v * NT + (size_t)B * n_vt * NT;
}

// Visual rows per relevance tile: the R of 128, 96 and 64 whose tiles give the
// busiest SM the fewest rows to take in (its tiles' visual and text rows,
// ceil(tiles / SMs) tiles), the larger R on a tie.
static int rel_tile_rows(int B, int N_v, int NT, int n_tb, int num_sms) {
  int best = kBM;
  long long best_cost = -1;
  for (int R = kBM; R >= 64; R -= 32) {
    const long long tiles = (long long)B * ((N_v + R - 1) / R) * n_tb;
    const long long cost = ((tiles + num_sms - 1) / num_sms) * (R + NT);
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best = R;
    }
  }
  return best;
}

// tiles and shared memory of the relevance
struct RelShape {
  int NTs, n_tb, NT, R, n_vt, n_stages;
  bool deep;    // one CTA per SM
  size_t smem;
};
constexpr size_t kRelSmemMax = 200 * 1024;
static RelShape rel_shape(int B, int N_v, int N_t_max, int num_sms) {
  RelShape h;
  h.NTs = rel_nt(N_t_max);
  h.n_tb = (h.NTs + kBM - 1) / kBM;  // text blocks, of equal rows but for the last
  h.NT = rel_nt((h.NTs + h.n_tb - 1) / h.n_tb);
  h.R = rel_tile_rows(B, N_v, h.NT, h.n_tb, num_sms);
  h.n_vt = (N_v + h.R - 1) / h.R;
  // one CTA per SM when the tiles do not fill the GPU or there are several text
  // blocks (deeper ring), else two
  // the MMA reads 128 A rows (16 KiB) from the start of a stage: the last
  // stage keeps that much room even when R + NT rows are fewer
  const size_t st_bytes = (size_t)(h.R + h.NT) * 128;
  const size_t tail = st_bytes > (size_t)kABytes ? 0 : (size_t)kABytes - st_bytes;
  h.deep = h.n_tb > 1 || (long long)B * h.n_vt <= num_sms;
  const size_t budget = (h.deep ? kRelSmemMax - 1024 : 110 * 1024 - 1024) - tail;
  const int ns = (int)(budget / st_bytes);
  h.n_stages = ns > kRelMaxStages ? kRelMaxStages : (ns < 2 ? 2 : ns);
  h.smem = (size_t)h.n_stages * st_bytes + tail + 1024;
  return h;
}

cudaError_t relevance_tc_launch(const SimArgs& a, const uint8_t* mask, const float* inv_t, float* inv_v,
                                float* p, float* ws, int num_sms, cudaStream_t s, cudaEvent_t mask_ready) {
  static std::atomic<bool> smem_set[64], smem_set2[64];  // per device, zero-initialised
  int dev = 0;
  cudaGetDevice(&dev);
  cudaError_t e = set_smem(relevance_fused_tc<false>, kRelSmemMax, &smem_set[dev < 64 ? dev : 0]);
  if (e == cudaSuccess) e = set_smem(relevance_fused_tc<true>, kRelSmemMax, &smem_set2[dev < 64 ? dev : 0]);
  if (e != cudaSuccess) return e;
  RelFusedArgs r;
  r.B = a.B;
  r.N_v = a.N_v;
  r.D = a.D;
  r.N_t_max = a.N_t_max;
  const RelShape h = rel_shape(a.B, a.N_v, a.N_t_max, num_sms);
  r.NTs = h.NTs;
  r.NT = h.NT;
  r.R = h.R;
  r.n_vt = h.n_vt;
  r.n_stages = h.n_stages;
  r.inv_t = inv_t;
  r.inv_v = inv_v;
  r.Y = ws;
  r.part = ws + (size_t)a.B * a.N_v * r.NTs;
  r.err = a.err;
  CUtensorMap mapV, mapT;
  if (make_tmap_bf16_2d(&mapV, a.emb_v, (uint64_t)a.B * a.N_v, (uint64_t)a.D, (uint64_t)a.D * 2, (uint32_t)r.R) ||
      make_tmap_bf16_2d(&mapT, a.emb_t, (uint64_t)a.B * a.N_t_max, (uint64_t)a.D, (uint64_t)a.D * 2,
                        (uint32_t)r.NT))
    return cudaErrorInvalidValue;
  e = h.n_tb == 1 ? launch_pdl(relevance_fused_tc<false>, dim3(r.n_vt, a.B), dim3(kThreads), h.smem, s, r, mapV, mapT)
                  : launch_pdl(relevance_fused_tc<true>, dim3(r.n_vt, a.B, h.n_tb), dim3(kRelLongThreads), h.smem, s, r, mapV, mapT);
  if (e != cudaSuccess) return e;
  const dim3 gf((a.N_v + 8 * kRelFinishRows - 1) / (8 * kRelFinishRows), a.B);
  const size_t smem_f = (size_t)r.NTs * (sizeof(float) + sizeof(int));
  if (mask_ready == nullptr) return launch_pdl(relevance_finish_kernel, gf, dim3(256), smem_f, s, r, a.text_len, mask, p);
  e = cudaStreamWaitEvent(s, mask_ready, 0);  // the first kernel that reads the mask
  if (e != cudaSuccess) return e;
  relevance_finish_kernel<<<gf, 256, smem_f, s>>>(r, a.text_len, mask, p);
  return cudaGetLastError();
}

}  // namespace provip

namespace provip {

// CTAs per tile and accumulators per CTA: 8 x 2 while the clusters fit the SMs at
// one CTA each, 4 x 4 beyond (the same 16 parts with fewer, longer CTAs); narrow
// embeddings with fewer K slices take the largest power of two of them.
static int crit_cluster(int B, int nt, int n_k, int num_sms) {
  int C = (long long)B * nt * nt * kCritMaxCluster <= num_sms ? kCritMaxCluster : kCritMaxAcc;
  while (C > n_k) C /= 2;
  return C;
}

constexpr size_t kCritTileBytes = (size_t)kBM * kCritLd * sizeof(float);
constexpr size_t kCritRingBytes = (size_t)kCritStages * kABytes;
constexpr size_t kCritWholeSmem = (kCritRingBytes > kCritTileBytes ? kCritRingBytes : kCritTileBytes) + 1024;

// Whether the critical rows, as one kernel, come first on the stream and the relevance
// follows instead of running beside them from another, without the events between.
// * Their CTAs take three quarters of the SMs or more: at 64 and 8 CTAs (8 anyres samples,
//   a video) the later start of the relevance costs more, 219 -> 223 us a pass and 178 ->
//   184, and at 80 to 112 it went either way.
// * The relevance takes at most two CTAs per SM at once: at 29 samples of 1440 rows (435
//   tiles) 292 -> 297 us and 277 -> 282, at 32 under 128 text rows 311 -> 320.
// * Where it takes one CTA per SM, on more than seven eighths of them, that CTA does not
//   fit beside one of the critical rows: where it does, it is put there and both run slower
//   than in turn. 15 and 16 samples of 576 rows under 32 and 64 text rows (135 and 144
//   tiles of 64 rows, rings of 98 and 128 KiB): 107 -> 115 us from a graph, 119 -> 119
//   launched one by one; 15 of width 2048 66 -> 72 and 72 -> 77, 29 of 300 rows (145) 120
//   -> 126 and 133 -> 133. On fewer SMs (102 to 128 tiles) it gains all the same: 19 samples
//   of 576 rows under 32 (114) 110..118 -> 106 and 123 -> 111.
// Elsewhere, over 15 to 38 samples of 300 to 1440 rows of widths 1024 to 5120, it gave 1 to
// 6%: 16 samples of 576 under 128 text rows 121 -> 119, 17 under 64 118 -> 112, 32 of width
// 5120 171 -> 167.
bool crit_leads(const SimArgs& a, int num_sms) {
  if (a.dtype != 1 || a.N_t_max > kBM || !relevance_tc_supported(a)) return false;
  if (4ll * a.B * crit_cluster(a.B, 1, (a.D + kBK - 1) / kBK, num_sms) < 3ll * num_sms) return false;
  const RelShape h = rel_shape(a.B, a.N_v, a.N_t_max, num_sms);
  const long long tiles = (long long)a.B * h.n_vt;
  if (!h.deep) return tiles <= 2ll * num_sms;
  // 228 KiB per SM; 8 KiB for both kernels' static parts and what a CTA reserves
  return 8 * tiles <= 7ll * num_sms || h.smem + kCritWholeSmem + 8 * 1024 > 228 * 1024;
}

cudaError_t crit_gram_tc_launch(const SimArgs& a, uint8_t* mask, float* r_out, float* G, int num_sms, bool* whole,
                                cudaStream_t s, bool early) {
  static std::atomic<bool> smem_set[64], smem_set2[64];  // per device, zero-initialised
  int dev = 0;
  cudaGetDevice(&dev);
  constexpr size_t smem1 = kCritWholeSmem, smem2 = (size_t)kCritStages * 2 * kABytes + 1024;
  static_assert(smem2 >= kCritTileBytes + 1024, "the tile part fits the stages");
  cudaError_t e = set_smem(crit_gram_tc<true>, smem1, &smem_set[dev < 64 ? dev : 0]);
  if (e == cudaSuccess) e = set_smem(crit_gram_tc<false>, smem2, &smem_set2[dev < 64 ? dev : 0]);
  if (e != cudaSuccess) return e;
  CUtensorMap mapT;
  if (make_tmap_bf16_2d(&mapT, a.emb_t, (uint64_t)a.B * a.N_t_max, (uint64_t)a.D, (uint64_t)a.D * 2, 128))
    return cudaErrorInvalidValue;
  CritArgs c;
  c.text_len = a.text_len;
  c.N_t_max = a.N_t_max;
  c.n_k = (a.D + kBK - 1) / kBK;
  c.nt = (a.N_t_max + kBM - 1) / kBM;
  c.G = G;
  c.mask = mask;
  c.r_out = r_out;
  c.err = a.err;
  *whole = c.nt == 1;
  c.early = early && *whole;
  const int C = crit_cluster(a.B, c.nt, c.n_k, num_sms);
  c.n_acc = C == kCritMaxCluster ? 2 : kCritMaxAcc;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3((unsigned)C, (unsigned)(c.nt * c.nt), (unsigned)a.B);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = *whole ? smem1 : smem2;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return *whole ? cudaLaunchKernelEx(&cfg, crit_gram_tc<true>, c, mapT)
                : cudaLaunchKernelEx(&cfg, crit_gram_tc<false>, c, mapT);
}

}  // namespace provip
