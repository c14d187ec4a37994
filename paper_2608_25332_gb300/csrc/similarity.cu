// Pre-LLM pass (Sec. 4.2-4.3), CUDA-core kernels.
//
//   crit_text:  G = E_t E_t^T (no scale), row softmax, r_j = mean_i R_ij,
//               T = { j : r_j > mean(r) } (all rows when none exceeds it).
//   relevance:  p_j = max_{i in T} ( cos(t_i, v_j) - mu_i ), where the row mean
//               mu_i = (1/N_v) sum_k cos(t_i, v_k) = <t_i / |t_i|, sum_k v_k / |v_k|> / N_v
//               is computed from the sum of the normalised visual rows, so the
//               |T| x N_v cosine matrix is never stored.
//   merge:      for each visual row j, the kept row of largest cosine
//               (= largest <v_j, v_k> / |v_k|, since |v_j| is common), ties to
//               the lower kept position; merged_a = mean of centroid a and its
//               members, summed in ascending row order.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "simt_split.cuh"

namespace provip {
namespace {

template <typename T>
__device__ __forceinline__ const T* row_ptr(const void* base, size_t row, int D) {
  return static_cast<const T*>(base) + row * (size_t)D;
}

// ---------------------------------------------------------------------------
// Sec. 4.2
// ---------------------------------------------------------------------------
// the fp32 text Gram: a cluster per 64 x 64 tile and part of K (simt_split.cuh;
// gridDim.z parts, each its own G), CTA c of it writing rows [c * 64 / C, ..)
__global__ void __launch_bounds__(split::kThreads, split::kCtasPerSm) crit_gram_kernel(const SimArgs a, int C, float* G) {
  extern __shared__ __align__(128) uint8_t ring[];
  __shared__ const float* arow[split::kTile];
  __shared__ const float* brow[split::kTile];
  const int rank = blockIdx.x % C, tile = blockIdx.x / C, b = blockIdx.y;
  const int nt = (a.N_t_max + split::kTile - 1) / split::kTile;
  const int r0 = tile / nt * split::kTile, c0 = tile % nt * split::kTile;
  int tl = a.text_len[b];
  if (tl < 0 || tl > a.N_t_max) tl = 0;
  if (r0 >= tl || c0 >= tl) return;  // every CTA of the cluster: nothing reads the tile
  if (threadIdx.x < split::kTile) {
    const int i = r0 + threadIdx.x, j = c0 + threadIdx.x;
    arow[threadIdx.x] = i < tl ? row_ptr<float>(a.emb_t, (size_t)b * a.N_t_max + i, a.D) : nullptr;
    brow[threadIdx.x] = j < tl ? row_ptr<float>(a.emb_t, (size_t)b * a.N_t_max + j, a.D) : nullptr;
  }
  __syncthreads();
  int k0, k1;
  split::share(a.D, blockIdx.z * C + rank, gridDim.z * C, k0, k1);
  split::tile_part<float>(arow, brow, k0, k1, ring, a.emb_t);
  G += (size_t)blockIdx.z * a.B * a.N_t_max * a.N_t_max;
  split::cluster_sync();
  const int n_rows = split::kTile / C, c = c0 + (threadIdx.x & 15) * 4;
  for (int i = threadIdx.x >> 4; i < n_rows; i += split::kThreads / 16) {
    const int r = rank * n_rows + i;
    const float4 g = split::sum_parts(ring, r, (threadIdx.x & 15) * 4, C);
    if (r0 + r >= tl) continue;
    float* o = G + ((size_t)b * a.N_t_max + r0 + r) * a.N_t_max + c;
    const float ge[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (c + e < tl) o[e] = ge[e];
  }
  split::cluster_sync();  // no CTA leaves while a peer may still read its part
}

// From the sample Grams G [B][Ntm][Ntm]: row softmax, column means r, threshold
// (the CUDA-core Gram's, and the tensor-core Gram's past 128 text rows). A cluster
// of kFinishCtas CTAs per sample, a row per warp at a time, the rows dealt to the
// warps of the cluster in turn: lane l takes columns l, l + 32, .., which stay in
// registers (kReg of them) up to 32 kReg text rows, else the row is read three
// times (from L1). A warp adds its rows' softmax per column, then the warps, then
// the CTAs are added in order. One CTA of 1024 threads per sample took 34 us for
// 300 text rows.
constexpr int kFinishCtas = 8;
constexpr int kCritMaxParts = 2;  // parts of K that the fp32 text Gram may leave to this kernel,
constexpr int kPartsReg = 4;      // for at most 32 * kPartsReg text rows
constexpr int kFinishWarps = 8;
constexpr size_t finish_smem(int N_t_max) { return (size_t)(kFinishWarps + 2) * N_t_max * sizeof(float); }
__device__ __forceinline__ void finish_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <int kReg>
__global__ void __launch_bounds__(32 * kFinishWarps) crit_finish_kernel(const SimArgs a, const float* G, int parts,
                                                                        uint8_t* mask, float* r_out) {
  extern __shared__ float sh[];  // part[kFinishWarps][Ntm], col[Ntm], rr[Ntm]
  float* col = sh + (size_t)kFinishWarps * a.N_t_max;
  float* rr = col + a.N_t_max;
  __shared__ float wsum[kFinishWarps];
  __shared__ int wcnt[kFinishWarps];
  const int rank = blockIdx.x, b = blockIdx.y;  // the cluster spans grid x
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int n = a.text_len[b];
  if (n < 0 || n > a.N_t_max) {
    if (rank == 0 && threadIdx.x == 0) set_error(a.err, kErrBadDeviceArg);
    n = 0;
  }
  const float* Gb = G + (size_t)b * a.N_t_max * a.N_t_max;
  float* part = sh + (size_t)warp * a.N_t_max;
  const int i0 = rank * kFinishWarps + warp;
  if constexpr (kReg > 0) {
    float acc[kReg];
#pragma unroll
    for (int q = 0; q < kReg; ++q) acc[q] = 0.f;
    for (int i = i0; i < n; i += kFinishCtas * kFinishWarps) {
      float v[kReg], m = -INFINITY, z = 0.f;
#pragma unroll
      for (int q = 0; q < kReg; ++q) v[q] = lane + 32 * q < n ? Gb[(size_t)i * a.N_t_max + lane + 32 * q] : 0.f;
      if constexpr (kReg <= kPartsReg) {
        float w[kCritMaxParts - 1][kReg];  // the further parts, added in order
#pragma unroll
        for (int p = 1; p < kCritMaxParts; ++p)
#pragma unroll
          for (int q = 0; q < kReg; ++q)
            w[p - 1][q] = p < parts && lane + 32 * q < n
                              ? Gb[((size_t)p * a.B * a.N_t_max + i) * a.N_t_max + lane + 32 * q] : 0.f;
#pragma unroll
        for (int p = 1; p < kCritMaxParts; ++p)
#pragma unroll
          for (int q = 0; q < kReg; ++q) v[q] += w[p - 1][q];
      }
#pragma unroll
      for (int q = 0; q < kReg; ++q)
        if (lane + 32 * q < n) m = fmaxf(m, v[q]);
      m = warp_max(m);
#pragma unroll
      for (int q = 0; q < kReg; ++q) {
        v[q] = lane + 32 * q < n ? expf(v[q] - m) : 0.f;
        z += v[q];
      }
      const float inv = 1.f / warp_sum(z);
#pragma unroll
      for (int q = 0; q < kReg; ++q) acc[q] += v[q] * inv;
    }
#pragma unroll
    for (int q = 0; q < kReg; ++q)
      if (lane + 32 * q < n) part[lane + 32 * q] = acc[q];
  } else {
    for (int j = lane; j < n; j += 32) part[j] = 0.f;
    for (int i = i0; i < n; i += kFinishCtas * kFinishWarps) {
      const float* row = Gb + (size_t)i * a.N_t_max;
      float m = -INFINITY, z = 0.f;
      for (int j = lane; j < n; j += 32) m = fmaxf(m, row[j]);
      m = warp_max(m);
      for (int j = lane; j < n; j += 32) z += expf(row[j] - m);
      const float inv = 1.f / warp_sum(z);
      for (int j = lane; j < n; j += 32) part[j] += expf(row[j] - m) * inv;
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kFinishWarps; ++w) s += sh[(size_t)w * a.N_t_max + j];
    col[j] = s;
  }
  finish_cluster_sync();  // every CTA's column sums
  if (rank == 0) {
    float pt = 0.f;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
      float s = 0.f;
#pragma unroll
      for (int q = 0; q < kFinishCtas; ++q) {
        uint32_t addr;
        float v;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(smem_u32(col + j)), "r"(q));
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
        s += v;
      }
      rr[j] = s / (float)n;
      pt += rr[j];
    }
    // mean(r), fixed-order block sum
    pt = warp_sum(pt);
    if (lane == 0) wsum[warp] = pt;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < kFinishWarps; ++w) tot += wsum[w];
    const float mean = n > 0 ? tot / (float)n : 0.f;
    int c = 0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) c += rr[j] > mean;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) wcnt[warp] = c;
    __syncthreads();
    int cnt = 0;
#pragma unroll
    for (int w = 0; w < kFinishWarps; ++w) cnt += wcnt[w];
    for (int j = threadIdx.x; j < a.N_t_max; j += blockDim.x) {
      const bool in = j < n && (cnt == 0 || rr[j] > mean);
      mask[(size_t)b * a.N_t_max + j] = in ? 1 : 0;
      if (r_out) r_out[(size_t)b * a.N_t_max + j] = j < n ? rr[j] : 0.f;
    }
  }
  finish_cluster_sync();  // no CTA leaves while CTA 0 may still read its column sums
}

// ---------------------------------------------------------------------------
// inverse row norms: one warp per row
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) inv_norm_kernel(const void* X, size_t rows, int D,
                                                       float* inv) {
  pdl_allow_next();  // a dependent reads inv only after this grid completes
  const size_t row = (size_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const T* p = static_cast<const T*>(X) + row * (size_t)D;
  float s = 0.f;
  for (int e = lane * 8; e < D; e += 256) {
    float v[8];
    load8(p + e, v);
#pragma unroll
    for (int q = 0; q < 8; ++q) s = fmaf(v[q], v[q], s);
  }
  s = warp_sum(s);
  if (lane == 0) inv[row] = s > 0.f ? 1.f / sqrtf(s) : 0.f;
  // completes after the kernel before it (the critical rows, when it runs beside them),
  // so that what waits for this grid finds that one's results too
  pdl_wait_prior();
}

// ---------------------------------------------------------------------------
// Sec. 4.3 relevance
// ---------------------------------------------------------------------------
// partial sums of normalised visual rows: part[z][b][d] over rows z*chunk..
// (8 rows in flight per step; the adds stay in row order)
template <typename T>
__global__ void __launch_bounds__(256) vis_sum_kernel(const SimArgs a, const float* inv_v,
                                                      float* part, int chunk) {
  const int d = blockIdx.x * 256 + threadIdx.x;
  const int b = blockIdx.y, z = blockIdx.z;
  if (d >= a.D) return;
  const int j0 = z * chunk, j1 = min(a.N_v, j0 + chunk);
  const T* E = static_cast<const T*>(a.emb_v) + (size_t)b * a.N_v * a.D;
  const float* iv = inv_v + (size_t)b * a.N_v;
  float s = 0.f;
  int j = j0;
  for (; j + 8 <= j1; j += 8) {
    float x[8], w[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      x[u] = to_f32(E[(size_t)(j + u) * a.D + d]);
      w[u] = iv[j + u];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) s = fmaf(x[u], w[u], s);
  }
  for (; j < j1; ++j) s = fmaf(to_f32(E[(size_t)j * a.D + d]), iv[j], s);
  part[((size_t)z * a.B + b) * a.D + d] = s;
}

// One read of the visual rows for both the inverse norms and the normalised
// sum: a CTA per (row chunk z, sample) fetches its rows kNormRows at a time
// with bulk copies (cp.async.bulk, one thread issuing) into shared memory;
// warp w takes row w's squared norm (lane-strided 16-byte pieces, then a warp
// sum) -> inv_v; then every thread adds its 16-byte pieces of the rows, in row
// order, scaled by their inverse norms -> part[z][b][d].
constexpr int kNormRows = 8;
constexpr int kNormThreads = 256;
constexpr int kNormMaxPieces = 4;  // 16-byte pieces per thread: D x esize <= 16 KiB
size_t norm_sum_smem(int D, int esize) { return (size_t)kNormRows * D * esize; }
bool norm_sum_supported(const SimArgs& a) {
  const int es = a.dtype == 0 ? 4 : 2;
  return (size_t)a.D * es <= (size_t)kNormMaxPieces * kNormThreads * 16 && (a.D * es) % 16 == 0;
}

// 8 bf16 of a shared-memory row as fp32 (plain shared load, not the read-only
// global path)
__device__ __forceinline__ void unpack8_shared(const uint8_t* p, float* o) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __bfloat1622float2(h[i]);
    o[2 * i] = f.x;
    o[2 * i + 1] = f.y;
  }
}

template <typename T>
__global__ void __launch_bounds__(kNormThreads) vis_norm_sum_kernel(const SimArgs a, float* inv_v,
                                                                    float* part, int chunk) {
  extern __shared__ __align__(128) uint8_t rows[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ float inv_s[kNormRows];
  constexpr int kVec = 16 / (int)sizeof(T);
  const int z = blockIdx.x, b = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = z * chunk, j1 = min(a.N_v, j0 + chunk);
  const T* E = static_cast<const T*>(a.emb_v) + (size_t)b * a.N_v * a.D;
  const uint32_t row_bytes = (uint32_t)a.D * (uint32_t)sizeof(T);
  const int n_pieces = (int)(row_bytes / 16);
  float acc[kNormMaxPieces][kVec];
#pragma unroll
  for (int k = 0; k < kNormMaxPieces; ++k)
#pragma unroll
    for (int e = 0; e < kVec; ++e) acc[k][e] = 0.f;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  uint32_t phase = 0;
  bool ok = true;
  for (int r0 = j0; r0 < j1; r0 += kNormRows) {
    const int nb = min(kNormRows, j1 - r0);
    if (threadIdx.x == 0) {
      const uint64_t pol = policy_evict_last();  // read again by the relevance Gram
      mbar_arrive_expect_tx(&bar, (uint32_t)nb * row_bytes);
      for (int q = 0; q < nb; ++q)
        bulk_g2s(rows + (size_t)q * row_bytes, E + (size_t)(r0 + q) * a.D, row_bytes, &bar, pol);
    }
    if (ok && !mbar_wait(&bar, phase, a.err)) ok = false;
    phase ^= 1u;
    if (warp < nb) {
      const uint8_t* row = rows + (size_t)warp * row_bytes;
      float sq = 0.f;
      for (int pc = lane; pc < n_pieces; pc += 32) {
        float v[8];
        if constexpr (sizeof(T) == 2) {
          unpack8_shared(row + (size_t)pc * 16, v);
#pragma unroll
          for (int q = 0; q < 8; ++q) sq = fmaf(v[q], v[q], sq);
        } else {
          const float4 f = *reinterpret_cast<const float4*>(row + (size_t)pc * 16);
          sq = fmaf(f.x, f.x, sq);
          sq = fmaf(f.y, f.y, sq);
          sq = fmaf(f.z, f.z, sq);
          sq = fmaf(f.w, f.w, sq);
        }
      }
      sq = warp_sum(sq);
      const float iv = sq > 0.f ? 1.f / sqrtf(sq) : 0.f;
      if (lane == 0) {
        inv_s[warp] = iv;
        inv_v[(size_t)b * a.N_v + r0 + warp] = iv;
      }
    }
    __syncthreads();
    for (int q = 0; q < nb; ++q) {
      const uint8_t* row = rows + (size_t)q * row_bytes;
      const float w = inv_s[q];
#pragma unroll
      for (int k = 0; k < kNormMaxPieces; ++k) {
        const int pc = k * kNormThreads + (int)threadIdx.x;
        if (pc >= n_pieces) continue;
        if constexpr (sizeof(T) == 2) {
          float v[8];
          unpack8_shared(row + (size_t)pc * 16, v);
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[k][e] = fmaf(v[e], w, acc[k][e]);
        } else {
          const float4 f = *reinterpret_cast<const float4*>(row + (size_t)pc * 16);
          acc[k][0] = fmaf(f.x, w, acc[k][0]);
          acc[k][1] = fmaf(f.y, w, acc[k][1]);
          acc[k][2] = fmaf(f.z, w, acc[k][2]);
          acc[k][3] = fmaf(f.w, w, acc[k][3]);
        }
      }
    }
    __syncthreads();  // the rows may be refilled
  }
  float* out = part + ((size_t)z * a.B + b) * a.D;
#pragma unroll
  for (int k = 0; k < kNormMaxPieces; ++k) {
    const int pc = k * kNormThreads + (int)threadIdx.x;
    if (pc >= n_pieces) continue;
#pragma unroll
    for (int e = 0; e < kVec; ++e) out[pc * kVec + e] = acc[k][e];
  }
}

// sum[b][d] = sum over the row chunks z of part[z][b][d] (fixed order)
__global__ void __launch_bounds__(256) vis_sum_reduce_kernel(const SimArgs a, const float* part,
                                                             int nz, float* sum) {
  const int d = blockIdx.x * 256 + threadIdx.x;
  const int b = blockIdx.y;
  if (d >= a.D) return;
  const float* p = part + (size_t)b * a.D + d;
  const size_t step = (size_t)a.B * a.D;
  float s = 0.f;
  for (int z0 = 0; z0 < nz; z0 += 32) {  // 32 loads in flight, the adds in chunk order
    float x[32];
#pragma unroll
    for (int u = 0; u < 32; ++u) x[u] = z0 + u < nz ? p[(size_t)(z0 + u) * step] : 0.f;
#pragma unroll
    for (int u = 0; u < 32; ++u)
      if (z0 + u < nz) s += x[u];
  }
  sum[(size_t)b * a.D + d] = s;
}

// mu_i and 1/|t_i| for the text rows (one warp per row, 8 elements per lane step)
template <typename T>
__global__ void __launch_bounds__(256) text_mu_kernel(const SimArgs a, const float* sum,
                                                      float* mu, float* invt) {
  const int b = blockIdx.y;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= a.N_t_max) return;
  const int tl = min(max(a.text_len[b], 0), a.N_t_max);
  if (i >= tl) {
    if (lane == 0) {
      mu[(size_t)b * a.N_t_max + i] = 0.f;
      invt[(size_t)b * a.N_t_max + i] = 0.f;
    }
    return;
  }
  const T* t = static_cast<const T*>(a.emb_t) + ((size_t)b * a.N_t_max + i) * a.D;
  const float* sv = sum + (size_t)b * a.D;
  float ss = 0.f, dt = 0.f;
#pragma unroll 4
  for (int d = lane * 8; d < a.D; d += 256) {
    float x[8];
    load8(t + d, x);
    const float4 s0 = *reinterpret_cast<const float4*>(sv + d);
    const float4 s1 = *reinterpret_cast<const float4*>(sv + d + 4);
    const float sw[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      ss = fmaf(x[q], x[q], ss);
      dt = fmaf(x[q], sw[q], dt);
    }
  }
  ss = warp_sum(ss);
  dt = warp_sum(dt);
  if (lane == 0) {
    const float iv = ss > 0.f ? 1.f / sqrtf(ss) : 0.f;
    invt[(size_t)b * a.N_t_max + i] = iv;
    mu[(size_t)b * a.N_t_max + i] = dt * iv / (float)a.N_v;
  }
}

// p_j = max over critical rows of cos - mu. A cluster per 64 visual rows takes the
// critical text rows (only those: their list is compacted first, kRelWin text
// rows at a time) in blocks of 64 (simt_split.cuh); CTA c of it adds and keeps the
// maxima of visual rows [c * 64 / C, ..).
constexpr int kRelWin = 1024;
template <typename T>
__global__ void __launch_bounds__(split::kThreads, split::kCtasPerSm) relevance_kernel(const SimArgs a, int C, const uint8_t* mask,
                                                                    const float* inv_v, const float* mu,
                                                                    const float* invt, float* p) {
  extern __shared__ __align__(128) uint8_t ring[];
  __shared__ const T* arow[split::kTile];
  __shared__ const T* brow[split::kTile];
  __shared__ uint16_t crit[kRelWin];
  __shared__ int wtot[split::kThreads / 32];
  __shared__ __align__(16) float4 red[split::kThreads];
  const int rank = blockIdx.x % C, b = blockIdx.y, c0 = blockIdx.x / C * split::kTile;
  const int tl = min(max(a.text_len[b], 0), a.N_t_max);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // this thread's four visual rows, and its text rows of a block: rgrp, rgrp + n_grp, ..
  const int nc = split::kTile / C, nq = nc / 4, n_grp = split::kThreads / nq;
  const int quad = tid % nq, rgrp = tid / nq;
  const int j0 = c0 + rank * nc + quad * 4;
  float iv[4], best[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    iv[e] = j0 + e < a.N_v ? inv_v[(size_t)b * a.N_v + j0 + e] : 0.f;
    best[e] = -INFINITY;
  }
  if (tid < split::kTile) {
    const int j = c0 + tid;
    brow[tid] = j < a.N_v ? row_ptr<T>(a.emb_v, (size_t)b * a.N_v + j, a.D) : nullptr;
  }
  int k0, k1;
  split::share(a.D, rank, C, k0, k1);
  for (int w0 = 0; w0 < tl; w0 += kRelWin) {
    int nT = 0;  // critical rows of the window
    for (int i0 = 0; i0 < kRelWin && w0 + i0 < tl; i0 += split::kThreads) {
      const int i = w0 + i0 + tid;
      const bool in = i < tl && mask[(size_t)b * a.N_t_max + i] != 0;
      const unsigned bal = __ballot_sync(0xffffffffu, in);
      if (lane == 0) wtot[warp] = __popc(bal);
      __syncthreads();
      int before = nT;
#pragma unroll
      for (int w = 0; w < split::kThreads / 32; ++w) {
        before += w < warp ? wtot[w] : 0;
        nT += wtot[w];
      }
      if (in) crit[before + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(i - w0);
      __syncthreads();
    }
    for (int r0 = 0; r0 < nT; r0 += split::kTile) {
      if (tid < split::kTile)
        arow[tid] = r0 + tid < nT
                        ? row_ptr<T>(a.emb_t, (size_t)b * a.N_t_max + w0 + crit[r0 + tid], a.D) : nullptr;
      __syncthreads();
      split::tile_part<T>(arow, brow, k0, k1, ring, a.emb_v);
      split::cluster_sync();
      for (int r = rgrp; r < min(split::kTile, nT - r0); r += n_grp) {
        const float4 v = split::sum_parts(ring, r, rank * nc + quad * 4, C);
        const size_t i = (size_t)b * a.N_t_max + w0 + crit[r0 + r];
        const float it = invt[i], m = mu[i];
        best[0] = fmaxf(best[0], v.x * it * iv[0] - m);
        best[1] = fmaxf(best[1], v.y * it * iv[1] - m);
        best[2] = fmaxf(best[2], v.z * it * iv[2] - m);
        best[3] = fmaxf(best[3], v.w * it * iv[3] - m);
      }
      split::cluster_sync();  // the parts have been read
    }
    __syncthreads();  // crit is rewritten by the next window
  }
  red[tid] = make_float4(best[0], best[1], best[2], best[3]);
  __syncthreads();
  if (rgrp == 0) {
    float4 m = red[quad];
    for (int g = 1; g < n_grp; ++g) {
      const float4 o = red[g * nq + quad];
      m.x = fmaxf(m.x, o.x);
      m.y = fmaxf(m.y, o.y);
      m.z = fmaxf(m.z, o.z);
      m.w = fmaxf(m.w, o.w);
    }
    const float me[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (j0 + e < a.N_v) p[(size_t)b * a.N_v + j0 + e] = me[e];
  }
}

// ---------------------------------------------------------------------------
// Sec. 4.3 merge
// ---------------------------------------------------------------------------
// Per sample (one CTA of 1024 threads): the kept-position map kpos[b][j] =
// a if j == keep[b][a], else -1, and the rows not kept in ascending order,
// pruned[b][0 .. cap) (ballot compaction), -1 past the last one. cap is N_v - keep, which a
// valid keep_idx fills, or N_v. With an invalid one (reported) more rows are not kept; those
// past cap are marked -2 in the map.
__global__ void __launch_bounds__(1024) merge_index_kernel(const int* keep_idx, int keep, int N_v, int* kpos,
                                                           int* pruned, int cap, unsigned* err) {
  __shared__ int warp_tot[32];
  const int b = blockIdx.x;
  int* kp = kpos + (size_t)b * N_v;
  const int* ki = keep_idx + (size_t)b * keep;
  for (int j = threadIdx.x; j < N_v; j += blockDim.x) kp[j] = -1;
  __syncthreads();
  for (int q = threadIdx.x; q < keep; q += blockDim.x) {
    const int j = ki[q];
    if (j < 0 || j >= N_v || (q > 0 && ki[q - 1] >= j)) {
      set_error(err, kErrBadDeviceArg);
      continue;
    }
    kp[j] = q;
  }
  __syncthreads();  // the map is complete (global writes of this block)
  int* out = pruned + (size_t)b * cap;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int base = 0;
  for (int j0 = 0; j0 < N_v; j0 += blockDim.x) {
    const int j = j0 + threadIdx.x;
    const bool pr = j < N_v && kp[j] < 0;
    const unsigned bal = __ballot_sync(0xffffffffu, pr);
    if (lane == 0) warp_tot[warp] = __popc(bal);
    __syncthreads();
    int off = 0, tot = 0;
    for (int w = 0; w < nw; ++w) {
      off += w < warp ? warp_tot[w] : 0;
      tot += warp_tot[w];
    }
    const int pos = base + off + __popc(bal & ((1u << lane) - 1u));
    if (pr && pos < cap) out[pos] = j;
    if (pr && pos >= cap) kp[j] = -2;
    base += tot;
    __syncthreads();
  }
  for (int i = base + (int)threadIdx.x; i < cap; i += blockDim.x) out[i] = -1;
}
__device__ __forceinline__ bool better(float v, int i, float bv, int bi) {
  return v > bv || (v == bv && i < bi);
}

// Argmax over one split of the kept columns for 64 pruned rows: a cluster per
// (row tile, split) walks the split's 64-column tiles (simt_split.cuh); CTA c of it
// adds rows [c * 64 / C, ..) and keeps their running (max, lowest position). The list of
// a sample has room for n_list rows, -1 past the last one.
template <typename T>
__global__ void __launch_bounds__(split::kThreads, split::kCtasPerSm) merge_argmax_kernel(const SimArgs a, int C, const int* pruned,
                                                                       int n_list, const int* keep_idx, int keep,
                                                                       const float* inv_v, int n_split,
                                                                       float* ws_best, int* ws_bidx) {
  extern __shared__ __align__(128) uint8_t ring[];
  __shared__ const T* arow[split::kTile];
  __shared__ const T* brow[split::kTile];
  __shared__ int rowj[split::kTile];
  __shared__ float kinv[split::kTile];
  const int rank = blockIdx.x % C, r0 = blockIdx.x / C * split::kTile, b = blockIdx.y, part = blockIdx.z;
  const int ntile = (keep + split::kTile - 1) / split::kTile;
  const int t0 = (int)((long long)ntile * part / n_split), t1 = (int)((long long)ntile * (part + 1) / n_split);
  const int tid = threadIdx.x, kg = tid & 15;
  if (tid < split::kTile) {
    const int j = r0 + tid < n_list ? pruned[(size_t)b * n_list + r0 + tid] : -1;
    const bool ok = j >= 0 && j < a.N_v;
    rowj[tid] = ok ? j : -1;
    arow[tid] = ok ? row_ptr<T>(a.emb_v, (size_t)b * a.N_v + j, a.D) : nullptr;
  }
  int k0, k1;
  split::share(a.D, rank, C, k0, k1);
  const int n_rows = split::kTile / C;
  constexpr int kAtOnce = split::kThreads / 16;  // rows a block takes at once
  constexpr int kRowsPer = split::kTile / kAtOnce;
  float bv[kRowsPer];
  int bi[kRowsPer];
#pragma unroll
  for (int u = 0; u < kRowsPer; ++u) {
    bv[u] = -INFINITY;
    bi[u] = 0x7fffffff;
  }
  for (int t = t0; t < t1; ++t) {
    const int a0 = t * split::kTile;
    if (tid < split::kTile) {
      const int j = a0 + tid < keep ? keep_idx[(size_t)b * keep + a0 + tid] : -1;
      const bool ok = j >= 0 && j < a.N_v;
      brow[tid] = ok ? row_ptr<T>(a.emb_v, (size_t)b * a.N_v + j, a.D) : nullptr;
      kinv[tid] = ok ? inv_v[(size_t)b * a.N_v + j] : 0.f;
    }
    __syncthreads();
    if (rowj[0] < 0) return;  // every CTA of the cluster: the list ends before the tile
    split::tile_part<T>(arow, brow, k0, k1, ring, a.emb_v);
    split::cluster_sync();
#pragma unroll
    for (int u = 0; u < kRowsPer; ++u) {
      if ((tid >> 4) + kAtOnce * u >= n_rows) continue;  // warp-uniform
      const float4 g = split::sum_parts(ring, rank * n_rows + (tid >> 4) + kAtOnce * u, kg * 4, C);
      const float ge[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int ap = a0 + kg * 4 + e;
        const float v = ge[e] * kinv[kg * 4 + e];
        if (ap < keep && better(v, ap, bv[u], bi[u])) {
          bv[u] = v;
          bi[u] = ap;
        }
      }
    }
    split::cluster_sync();  // the parts and kinv have been read
  }
  // combine the 16 lanes of each row
#pragma unroll
  for (int u = 0; u < kRowsPer; ++u) {
    if ((tid >> 4) + kAtOnce * u >= n_rows) continue;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv[u], o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi[u], o);
      if (better(ov, oi, bv[u], bi[u])) {
        bv[u] = ov;
        bi[u] = oi;
      }
    }
    const int j = rowj[rank * n_rows + (tid >> 4) + kAtOnce * u];
    if (kg == 0 && j >= 0) {
      ws_best[((size_t)part * a.B + b) * a.N_v + j] = bv[u];
      ws_bidx[((size_t)part * a.B + b) * a.N_v + j] = bi[u];
    }
  }
}

// assign[b][j]: own position for kept rows, best over splits for the others
// (and clears *n_long, the counter of the sort that follows, when given)
__global__ void merge_assign_kernel(const SimArgs a, const int* kpos, int n_split,
                                    const float* ws_best, const int* ws_bidx, int* assign, int* n_long) {
  pdl_wait_prior();  // the partials come from the Gram before
  pdl_allow_next();
  if (n_long != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *n_long = 0;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)a.B * a.N_v) return;
  const int kp = kpos[i];
  if (kp != -1) {
    assign[i] = max(kp, 0);  // -2: a row that an invalid keep_idx left out of the pruned list
    return;
  }
  float bv = -INFINITY;
  int bi = 0x7fffffff;
  for (int s = 0; s < n_split; ++s) {
    const float v = ws_best[(size_t)s * a.B * a.N_v + i];
    const int ix = ws_bidx[(size_t)s * a.B * a.N_v + i];
    if (better(v, ix, bv, bi)) {
      bv = v;
      bi = ix;
    }
  }
  // a zero or non-finite row compares equal everywhere: lowest position
  assign[i] = bi == 0x7fffffff ? 0 : bi;
}

// merged[b][a] = (sum of rows j with assign[b][j] == a, ascending j) / count.
// The member lists come from a counting sort per sample: counts (atomics),
// exclusive offsets, unordered fill, and a list of the centroids with more than
// kMeanShort members (n_long of them over the batch, in no particular order).
// A task is a column slice of 128 16-byte pieces, one per thread (a column's sum
// needs no other column), of kMeanGroup consecutive centroids: their member lists
// are one contiguous run, ordered within each centroid by rank (ascending row index,
// so the sum order is fixed) into one list of rows, and every thread streams its
// piece of those rows kMeanDeep copies ahead (cp.async) through its own
// shared-memory slots, with no block barrier between rows, closing a centroid's
// mean where its last row passes. The index chain (offsets, members, ranks) is paid
// once for the group, and the loads run on across its centroids. With a CTA per
// centroid, its whole rows fetched three at a time, 576 centroids of 32 samples of
// width 5120 took 56 us (240 MB, 4.3 TB/s), 2304 of one sample 31 us, and take 45 us
// (5.3 TB/s) and 25 us; groups of 16 and of 4 were within 2% or slower.
// Centroids with more than kMeanShort members (background that many tokens
// resemble) would hold a group's CTA while the GPU drains, so the grid's first CTAs
// take them, a slice of one centroid each, their members put in ascending order by
// rank or, where there are many, by a bitmap over windows of kMeanWin rows. With
// every list in one CTA, a bf16 batch of 8 x 2880 rows whose largest centroids gather
// some hundreds took 143 us here where the 253 MB it moves take 37.
constexpr int kMeanShort = 16;  // members of a centroid that a group's CTA takes
constexpr int kMeanGroup = 8;   // centroids of a group
constexpr int kMeanDeep = 12;   // pieces in flight per thread
constexpr int kMeanRank = 256;  // members of a long centroid that are ordered by rank
constexpr int kMeanWin = 1024;
constexpr int kMeanThreads = 128;
constexpr size_t kMeanSmem = (size_t)kMeanDeep * kMeanThreads * 16;
// centroids whose counters the sort keeps in shared memory: 8 bytes each beside the
// warps' totals, in the 48 KiB that a kernel has without an attribute
constexpr int kSortWarps = 32;
constexpr int kSortSmemKeep = (48 * 1024 - kSortWarps * (int)sizeof(int)) / (2 * (int)sizeof(int));

// Counting sort of one sample's rows by centroid (one CTA of 1024 threads):
// count[b][a] = rows assigned to a, offset[b][.] its exclusive scan, and
// members[b][offset[a] ..] the rows of a in no particular order (the means
// rank them), and b * keep + a of every centroid with more than kMeanShort rows
// appended to long_list (*n_long entries over the batch). The block-wide barriers
// order the phases (global memory of this block only). Bound by latency: with a row's
// load and atomic at a time and a barriered scan per 1024 centroids, the pass of a
// video (9216 rows, 2304 centroids, one CTA) took 183 us, now 181.
template <bool kSmem>
__global__ void __launch_bounds__(1024) merge_sort_kernel(const int* assign, int N_v, int keep, int* count,
                                                          int* offset, int* cursor, int* members, int* n_long,
                                                          int* long_list) {
  extern __shared__ int sort_sm[];  // kSmem: counts [keep], then offsets / cursors [keep]
  __shared__ int warp_tot[kSortWarps];
  pdl_wait_prior();  // the assignment comes from the kernel before
  pdl_allow_next();
  const int b = blockIdx.x;
  const int* as = assign + (size_t)b * N_v;
  int* cnt_g = count + (size_t)b * keep;
  int* off_g = offset + (size_t)b * keep;
  // the counters: shared memory for at most kSortSmemKeep centroids, else the
  // global scratch (cursor)
  int* cnt = kSmem ? sort_sm : cnt_g;
  int* cur = kSmem ? sort_sm + keep : cursor + (size_t)b * keep;
  for (int q = threadIdx.x; q < keep; q += blockDim.x) {
    cnt[q] = 0;
    cur[q] = 0;
  }
  __syncthreads();
  // four rows of a thread at a time, their loads and their atomics in flight together
  for (int j0 = threadIdx.x; j0 < N_v; j0 += 4096) {
    int ap[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) ap[u] = j0 + 1024 * u < N_v ? as[j0 + 1024 * u] : -1;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (ap[u] >= 0 && ap[u] < keep) atomicAdd(&cnt[ap[u]], 1);
  }
  __syncthreads();
  // the exclusive scan, a run of consecutive centroids per thread
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (keep + 1023) / 1024, a0 = (int)threadIdx.x * per, a1 = min(a0 + per, keep);
  int sum = 0;
  for (int ap = a0; ap < a1; ++ap) sum += cnt[ap];
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  // the warps before this one: every warp adds their totals itself
  int o = lane < warp ? warp_tot[lane] : 0;
#pragma unroll
  for (int sh = 16; sh > 0; sh >>= 1) o += __shfl_xor_sync(0xffffffffu, o, sh);
  o += incl - sum;
  for (int ap = a0; ap < a1; ++ap) {
    const int v = cnt[ap];
    off_g[ap] = o;
    if (v > kMeanShort) long_list[atomicAdd(n_long, 1)] = b * keep + ap;
    if (kSmem) {
      cnt_g[ap] = v;
      cur[ap] = o;  // the fill's running position
    }
    o += v;
  }
  __syncthreads();
  for (int j0 = threadIdx.x; j0 < N_v; j0 += 4096) {
    int ap[4], pos[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) ap[u] = j0 + 1024 * u < N_v ? as[j0 + 1024 * u] : -1;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (ap[u] < 0 || ap[u] >= keep) continue;
      pos[u] = kSmem ? atomicAdd(&cur[ap[u]], 1) : off_g[ap[u]] + atomicAdd(&cur[ap[u]], 1);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (ap[u] >= 0 && ap[u] < keep) members[(size_t)b * N_v + pos[u]] = j0 + 1024 * u;
  }
}

// the addition of 16 raw bytes of a row to Acc values (8 bf16 or 4 fp32)
__device__ __forceinline__ void add16(float* acc, const uint4& u, const __nv_bfloat16*) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __bfloat1622float2(h[i]);
    acc[2 * i] += f.x;
    acc[2 * i + 1] += f.y;
  }
}
__device__ __forceinline__ void add16(double* acc, const uint4& u, const float*) {
  acc[0] += (double)__uint_as_float(u.x);
  acc[1] += (double)__uint_as_float(u.y);
  acc[2] += (double)__uint_as_float(u.z);
  acc[3] += (double)__uint_as_float(u.w);
}
// The running sum of fp32 values as an unevaluated hi + mid + lo: the rounding error of
// every addition to hi is recovered exactly (Knuth's TwoSum) and added to mid, that
// addition's error to lo. lo itself is rounded, and settle(), every 256 rows, keeps it
// below an ulp of mid, so n rows are added to within n 2^-56 of the largest partial
// sum, where double allows n 2^-53; and acc_mean rounds the quotient once. Sums of
// 1 to 9000 rows, spread over 2^60, cancelling or subnormal, were all correctly
// rounded; in double 1 in 500 of those that cancel to 1e-7 of their largest partial
// were not, and as pairs of floats 1 in 4. The GPU adds 128 floats per SM clock but
// only two doubles: in double, with a division per element, the means of one fp32 image
// (576 rows of 4096) took 66 us; as pairs they took 14, as triples 16 (the pass 105.4 with
// either), and the merge of 16 such images 314 and 322. A sum that leaves fp32's
// range or meets an infinity or a NaN is taken again in double.
struct Sum3 {
  float hi, mid, lo;
};
// a + b = the returned sum + e, exactly
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float t = a + b, z = t - a;
  e = (a - (t - z)) + (b - z);
  return t;
}
__device__ __forceinline__ void add1(Sum3& s, float x) {
  float e, f;
  s.hi = two_sum(s.hi, x, e);
  s.mid = two_sum(s.mid, e, f);
  s.lo += f;
}
__device__ __forceinline__ void add16(Sum3* acc, const uint4& u, const float*) {
  add1(acc[0], __uint_as_float(u.x));
  add1(acc[1], __uint_as_float(u.y));
  add1(acc[2], __uint_as_float(u.z));
  add1(acc[3], __uint_as_float(u.w));
}
constexpr int kSettleRows = 256;
__device__ __forceinline__ void settle(float&) {}
__device__ __forceinline__ void settle(double&) {}
__device__ __forceinline__ void settle(Sum3& s) {
  float e;
  s.hi = two_sum(s.hi, s.mid, e);
  s.mid = two_sum(e, s.lo, s.lo);
  s.hi = two_sum(s.hi, s.mid, s.mid);
  s.mid = two_sum(s.mid, s.lo, s.lo);
}
__device__ __forceinline__ void acc_zero(float& a) { a = 0.f; }
__device__ __forceinline__ void acc_zero(double& a) { a = 0.0; }
__device__ __forceinline__ void acc_zero(Sum3& a) { a.hi = a.mid = a.lo = 0.f; }
// sum / n; a triple that is not finite clears ok
__device__ __forceinline__ float acc_mean(float a, int n, bool&) { return a / (float)n; }
__device__ __forceinline__ float acc_mean(double a, int n, bool&) { return (float)(a / (double)n); }
__device__ __forceinline__ float acc_mean(Sum3 a, int n, bool& ok) {
  if (!(fabsf(a.hi) <= 3.0e38f && fabsf(a.mid) <= 3.0e38f && fabsf(a.lo) <= 3.0e38f)) ok = false;
  settle(a);
  if (!(fabsf(a.hi) >= 0x1p-90f)) {  // the remainders below could be subnormal
    return a.hi == 0.f ? 0.f : (float)(((double)a.hi + (double)a.mid + (double)a.lo) / (double)n);
  }
  // q, the quotient of hi to about an ulp; c, of what q leaves (an exact remainder, as
  // n < 2^22) and of mid; d, of what both leave
  const float fn = (float)n, inv = 1.f / fn, q = a.hi * inv;
  float t, e;
  const float r = two_sum(fmaf(-q, fn, a.hi), a.mid, t), c = r * inv;
  const float d = (fmaf(-c, fn, r) + (t + a.lo)) * inv;
  // c + d rounded to odd, so that q + (c + d), rounded to nearest, is rounded only once
  const float u = two_sum(c, d, e);
  int bits = __float_as_int(u);
  if (e != 0.f && (bits & 1) == 0) bits += (e > 0.f) == (u > 0.f) ? 1 : -1;
  return q + __int_as_float(bits);
}
// 16 bytes of a row from fp32 values, rounded to nearest even
__device__ __forceinline__ void store16(__nv_bfloat16* p, const float* v) {
  uint4 u;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
  *reinterpret_cast<uint4*>(p) = u;
}
__device__ __forceinline__ void store16(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Column slice `slice` (a 16-byte piece per thread) of centroid `cen` = b * keep
// + a, whose n members lie unordered at mem[0..n). ring: kMeanDeep pieces per
// thread. Called by every thread of the block; false where a thread's sums are to
// be taken again in a wider type.
template <typename T, typename Acc>
__device__ __forceinline__ bool mean_long(const SimArgs& a, int b, int n, const int* mem, int slice, uint4* ring,
                                          uint32_t* bits, int* pre, uint16_t* list, T* out) {
  constexpr int kVec = 16 / (int)sizeof(T);
  const int pc = slice * kMeanThreads + (int)threadIdx.x;
  const bool has = pc < a.D / kVec;
  const T* E = static_cast<const T*>(a.emb_v) + (size_t)b * a.N_v * a.D + (size_t)(has ? pc : 0) * kVec;
  uint4* mine = ring + threadIdx.x;
  Acc acc[kVec];
#pragma unroll
  for (int e = 0; e < kVec; ++e) acc_zero(acc[e]);
  // adds rows at[0..cnt) of base in order
  auto stream = [&](const T* base, const auto* at, int cnt) {
    // one group per row, empty past the last, so that a fixed count is in flight
    auto fetch = [&](int i) {
      if (has && i < cnt) cp_async16(mine + (i % kMeanDeep) * kMeanThreads, base + (size_t)at[i] * a.D);
      cp_async_commit();
    };
#pragma unroll 1
    for (int i = 0; i < kMeanDeep - 1; ++i) fetch(i);
#pragma unroll 1
    for (int i = 0; i < cnt; ++i) {
      fetch(i + kMeanDeep - 1);
      cp_async_wait<kMeanDeep - 1>();
      if (has) add16(acc, mine[(i % kMeanDeep) * kMeanThreads], E);
      if ((i + 1) % kSettleRows == 0)
#pragma unroll
        for (int e = 0; e < kVec; ++e) settle(acc[e]);
    }
#pragma unroll
    for (int e = 0; e < kVec; ++e) settle(acc[e]);
    cp_async_wait<0>();
  };
  if (n <= kMeanRank) {
    int* un = reinterpret_cast<int*>(list);
    int* sorted = un + kMeanRank;
    const int n4 = (n + 3) / 4;
    __syncthreads();  // the previous task's list has been read
    for (int m = threadIdx.x; m < 4 * n4; m += kMeanThreads) un[m] = m < n ? mem[m] : 0x7fffffff;
    __syncthreads();
    for (int m = threadIdx.x; m < n; m += kMeanThreads) {
      const int v = un[m];
      int rank = 0;  // the number of smaller row indices (they are distinct)
      for (int q = 0; q < n4; ++q) {
        const int4 x = reinterpret_cast<const int4*>(un)[q];
        rank += (x.x < v) + (x.y < v) + (x.z < v) + (x.w < v);
      }
      sorted[rank] = v;
    }
    __syncthreads();
    stream(E, sorted, n);
  }
  for (int w0 = 0; n > kMeanRank && w0 < a.N_v; w0 += kMeanWin) {
    __syncthreads();  // the previous window's list has been read
    if (threadIdx.x < kMeanWin / 32) bits[threadIdx.x] = 0u;
    __syncthreads();
    for (int m = threadIdx.x; m < n; m += kMeanThreads) {
      const int j = mem[m] - w0;
      if (j >= 0 && j < kMeanWin) atomicOr(&bits[j >> 5], 1u << (j & 31));
    }
    __syncthreads();
    if (threadIdx.x < kMeanWin / 32) {  // warp 0: members before each word
      const int own = __popc(bits[threadIdx.x]);
      int incl = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)threadIdx.x >= o) incl += y;
      }
      pre[threadIdx.x] = incl - own;
      if (threadIdx.x == 31) pre[32] = incl;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < kMeanWin; j += kMeanThreads) {
      const uint32_t w = bits[j >> 5];
      if (w >> (j & 31) & 1u) list[pre[j >> 5] + __popc(w & ((1u << (j & 31)) - 1u))] = (uint16_t)j;
    }
    __syncthreads();
    const int cnt = pre[32];
    stream(E + (size_t)w0 * a.D, list, cnt);
  }
  bool ok = true;
  if (has) {
    float v[kVec];
#pragma unroll
    for (int e = 0; e < kVec; ++e) v[e] = acc_mean(acc[e], n, ok);
    store16(out + (size_t)pc * kVec, v);
  }
  return ok;
}

template <typename T, typename Acc>
__global__ void __launch_bounds__(kMeanThreads, 8)
    merge_mean_kernel(const SimArgs a, const int* count, const int* offset, const int* members_all, int keep,
                      void* merged, const int* n_long, const int* long_list, int long_ctas) {
  static_assert(kMeanWin / 32 == 32, "a word of the window per lane");
  static_assert(2 * kMeanRank * sizeof(int) <= kMeanWin * sizeof(uint16_t), "the ranked lists take the window's place");
  static_assert(kMeanGroup * kMeanShort == kMeanThreads, "a member of the group per thread");
  extern __shared__ __align__(128) uint4 mean_ring[];  // kMeanDeep pieces per thread
  __shared__ uint32_t bits[kMeanWin / 32];
  __shared__ int pre[kMeanWin / 32 + 1];
  __shared__ __align__(16) uint16_t list[kMeanWin];
  __shared__ int unsorted[kMeanThreads], rows[kMeanThreads];
  __shared__ int gcount[kMeanGroup], gstart[kMeanGroup + 1];
  __shared__ bool gbrief[kMeanGroup];
  constexpr int kVec = 16 / (int)sizeof(T);  // elements per 16-byte piece
  const int n_slices = (a.D / kVec + kMeanThreads - 1) / kMeanThreads;
  const int tid = threadIdx.x;
  pdl_wait_prior();  // the member lists come from the sort before
  if ((int)blockIdx.x < long_ctas) {
    const long long n_tasks = (long long)*n_long * n_slices;
    for (long long t = blockIdx.x; t < n_tasks; t += long_ctas) {
      const int cen = long_list[t / n_slices], b = cen / keep, n = count[cen];
      const int* mem = members_all + (size_t)b * a.N_v + offset[cen];
      T* out = static_cast<T*>(merged) + (size_t)cen * a.D;
      const bool ok = mean_long<T, Acc>(a, b, n, mem, (int)(t % n_slices), mean_ring, bits, pre, list, out);
      if constexpr (sizeof(T) == 4)
        if (__syncthreads_or(!ok))
          mean_long<T, double>(a, b, n, mem, (int)(t % n_slices), mean_ring, bits, pre, list, out);
    }
    return;
  }
  const int n_groups = (keep + kMeanGroup - 1) / kMeanGroup;
  const int task = (int)blockIdx.x - long_ctas;
  const int slice = task % n_slices, grp = task / n_slices;
  const int b = grp / n_groups, a0 = (grp - b * n_groups) * kMeanGroup, ng = min(kMeanGroup, keep - a0);
  const size_t cen0 = (size_t)b * keep + a0;
  // this thread's slot of the group: member q of its centroid g (as many slots as a
  // short centroid may have members); counts and offsets arrive together
  const int g = tid / kMeanShort, q = tid % kMeanShort;
  const int n_g = g < ng ? count[cen0 + g] : 0, off_g = g < ng ? offset[cen0 + g] : 0;
  const bool brief = n_g <= kMeanShort;  // the others are among the long ones
  const int v = brief && q < n_g ? members_all[(size_t)b * a.N_v + off_g + q] : 0x7fffffff;
  unsorted[tid] = v;
  if (q == 0) {
    gcount[g] = brief ? n_g : 0;
    gbrief[g] = brief;
  }
  __syncthreads();
  int before = 0;  // rows of the group's earlier centroids
#pragma unroll
  for (int h = 0; h < kMeanGroup; ++h) before += h < g ? gcount[h] : 0;
  if (brief && q < n_g) {
    int rank = 0;  // the number of smaller row indices (they are distinct)
#pragma unroll
    for (int h = 0; h < kMeanShort; ++h) rank += unsorted[g * kMeanShort + h] < v;
    rows[before + rank] = v;
  }
  if (q == 0) {
    gstart[g] = before;
    if (g == kMeanGroup - 1) gstart[kMeanGroup] = before + gcount[g];
  }
  __syncthreads();
  const int n_rows = gstart[kMeanGroup];
  const int pc = slice * kMeanThreads + tid;
  if (pc >= a.D / kVec) return;  // no barrier follows
  const T* E = static_cast<const T*>(a.emb_v) + (size_t)b * a.N_v * a.D + (size_t)pc * kVec;
  T* out = static_cast<T*>(merged) + cen0 * a.D + (size_t)pc * kVec;
  uint4* mine = mean_ring + tid;
  // one group per row, empty past the last, so that a fixed count is in flight
  auto fetch = [&](int i) {
    if (i < n_rows) cp_async16(mine + (i % kMeanDeep) * kMeanThreads, E + (size_t)rows[i] * a.D);
    cp_async_commit();
  };
#pragma unroll 1
  for (int i = 0; i < kMeanDeep - 1; ++i) fetch(i);
  int i = 0;
#pragma unroll 1
  for (int c = 0; c < ng; ++c) {
    const int end = gstart[c + 1], n = end - i;
    if (!gbrief[c]) continue;  // among the long ones
    Acc acc[kVec];
#pragma unroll
    for (int e = 0; e < kVec; ++e) acc_zero(acc[e]);
#pragma unroll 1
    for (; i < end; ++i) {
      fetch(i + kMeanDeep - 1);
      cp_async_wait<kMeanDeep - 1>();
      add16(acc, mine[(i % kMeanDeep) * kMeanThreads], E);
    }
    float m[kVec];
    bool fine = true;
#pragma unroll
    for (int e = 0; e < kVec; ++e) m[e] = n > 0 ? acc_mean(acc[e], n, fine) : 0.f;
    if constexpr (sizeof(T) == 4) {
      if (!fine) {
        double d[kVec];
#pragma unroll
        for (int e = 0; e < kVec; ++e) d[e] = 0.0;
        for (int r = end - n; r < end; ++r) add16(d, *reinterpret_cast<const uint4*>(E + (size_t)rows[r] * a.D), E);
#pragma unroll
        for (int e = 0; e < kVec; ++e) m[e] = acc_mean(d[e], n, fine);
      }
    }
    store16(out + (size_t)c * a.D, m);
  }
  cp_async_wait<0>();
}

}  // namespace

cudaError_t crit_text_launch(const SimArgs& a, uint8_t* mask, float* r_out, float* G, int num_sms,
                             cudaStream_t s, bool early) {
  int parts = 1;
  if (a.dtype == 0) {
    const int nt = (a.N_t_max + split::kTile - 1) / split::kTile;
    const int C = split::cluster_size((long long)a.B * nt * nt, a.D, num_sms);
    // where the largest clusters leave SMs idle, K in two parts, by the clusters' own rule
    // (at least 1024 elements a part) and where G's region holds them: the relevance of one
    // image waits for its 64 x 64 Gram over 4096 elements, and the pass went from 104.7 to
    // 98.5 us (four parts: the same, the relevance no longer waits)
    while (C == split::kMaxCluster && a.N_t_max <= 32 * kPartsReg &&
           2 * parts <= std::min(kCritMaxParts, crit_gram_parts(a.N_t_max, a.D)) &&
           2ll * parts * C * a.B * nt * nt <= (long long)split::kCtasPerSm * num_sms &&
           a.D / (2 * parts * C) >= 4 * split::kKT)
      parts *= 2;
    static std::atomic<bool> set[64];  // per device, zero-initialised
    const cudaError_t e = split::launch(crit_gram_kernel, split::kSmem<float>, set, dim3((unsigned)(C * nt * nt), (unsigned)a.B, (unsigned)parts), C, s, a, C, G);
    if (e != cudaSuccess) return e;
  } else {
    bool whole = false;
    cudaError_t e = crit_gram_tc_launch(a, mask, r_out, G, num_sms, &whole, s, early);
    if (e != cudaSuccess || whole) return e;
  }
  static std::atomic<bool> configured[64];  // per device, zero-initialised
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !configured[dev]) {
    cudaError_t e = cudaFuncSetAttribute(crit_finish_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)finish_smem(kCritMaxNt));
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3(kFinishCtas, (unsigned)a.B);
  cfg.blockDim = dim3(32 * kFinishWarps);
  cfg.dynamicSmemBytes = finish_smem(a.N_t_max);
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kFinishCtas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (a.N_t_max <= 32 * 4) return cudaLaunchKernelEx(&cfg, crit_finish_kernel<4>, a, G, parts, mask, r_out);
  if (a.N_t_max <= 32 * 16) return cudaLaunchKernelEx(&cfg, crit_finish_kernel<16>, a, G, parts, mask, r_out);
  return cudaLaunchKernelEx(&cfg, crit_finish_kernel<0>, a, G, parts, mask, r_out);
}

// 1/|e_j| (0 for a zero row) of the kept rows j = keep_idx[b][q] only, into
// inv_v[b][j] (the merge reads no other): a warp per row; an index out of range
// is reported and skipped.
template <typename T>
__global__ void __launch_bounds__(256) kept_inv_norm_kernel(const void* X, const int* keep_idx, int keep,
                                                            int N_v, int D, size_t rows, float* inv_v,
                                                            unsigned* err) {
  const size_t row = (size_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const size_t b = row / (size_t)keep;
  const int j = keep_idx[row];
  if (j < 0 || j >= N_v) {
    if (lane == 0) set_error(err, kErrBadDeviceArg);
    return;
  }
  const T* p = static_cast<const T*>(X) + (b * (size_t)N_v + (size_t)j) * (size_t)D;
  float s = 0.f;
  for (int e = lane * 8; e < D; e += 256) {
    float v[8];
    load8(p + e, v);
#pragma unroll
    for (int q = 0; q < 8; ++q) s = fmaf(v[q], v[q], s);
  }
  s = warp_sum(s);
  if (lane == 0) inv_v[b * (size_t)N_v + (size_t)j] = s > 0.f ? 1.f / sqrtf(s) : 0.f;
}

cudaError_t kept_inv_norm_launch(const SimArgs& a, const int* keep_idx, int keep, float* inv_v,
                                 cudaStream_t s) {
  const size_t rows = (size_t)a.B * keep;
  const unsigned grid = (unsigned)((rows + 7) / 8);
  if (a.dtype == 0)
    kept_inv_norm_kernel<float><<<grid, 256, 0, s>>>(a.emb_v, keep_idx, keep, a.N_v, a.D, rows, inv_v, a.err);
  else
    kept_inv_norm_kernel<__nv_bfloat16><<<grid, 256, 0, s>>>(a.emb_v, keep_idx, keep, a.N_v, a.D, rows, inv_v,
                                                            a.err);
  return cudaGetLastError();
}

cudaError_t vis_inv_norm_launch(const SimArgs& a, float* inv_v, cudaStream_t s) {
  const size_t rows = (size_t)a.B * a.N_v;
  const unsigned grid = (unsigned)((rows + 7) / 8);
  if (a.dtype == 0)
    inv_norm_kernel<float><<<grid, 256, 0, s>>>(a.emb_v, rows, a.D, inv_v);
  else
    inv_norm_kernel<__nv_bfloat16><<<grid, 256, 0, s>>>(a.emb_v, rows, a.D, inv_v);
  return cudaGetLastError();
}

cudaError_t relevance_launch(const SimArgs& a, const uint8_t* mask, float* inv_v, float* p,
                             float* ws_sum, float* ws_mu, float* ws_invt, int n_split,
                             int num_sms, cudaStream_t s, cudaEvent_t mask_ready, bool after_crit) {
  // bf16 (up to 4096 text rows): the text rows' inverse norms, one
  // tensor-core read of the visual rows (norms, cosines and de-meaning sums)
  // and a small max kernel
  if (relevance_tc_supported(a)) {
    const size_t rows = (size_t)a.B * a.N_t_max;
    if (after_crit) {
      const cudaError_t e = launch_pdl(inv_norm_kernel<__nv_bfloat16>, dim3((unsigned)((rows + 7) / 8)), dim3(256), 0,
                                       s, a.emb_t, rows, a.D, ws_invt);
      if (e != cudaSuccess) return e;
    } else {
      inv_norm_kernel<__nv_bfloat16><<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(a.emb_t, rows, a.D, ws_invt);
    }
    return relevance_tc_launch(a, mask, ws_invt, inv_v, p, ws_sum, num_sms, s, mask_ready);
  }
  const int chunk = (a.N_v + n_split - 1) / n_split;
  dim3 g1((a.D + 255) / 256, a.B, n_split);
  dim3 g2((a.N_t_max + 7) / 8, a.B);
  const int n_vt = (a.N_v + split::kTile - 1) / split::kTile;
  const int C = split::cluster_size((long long)a.B * n_vt, a.D, num_sms);
  const dim3 g3((unsigned)(C * n_vt), (unsigned)a.B);
  // ws_sum holds n_split partial sums followed by their total
  float* total = ws_sum + (size_t)n_split * a.B * a.D;
  dim3 g4((a.D + 255) / 256, a.B);
  // the inverse norms of the visual rows and their normalised sum, in one read
  // where the rows fit the shared-memory batch, else in two passes
  const bool fused = norm_sum_supported(a);
  if (fused) {
    static std::atomic<bool> configured[64];  // per device, zero-initialised
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !configured[dev]) {
      const int lim = kNormMaxPieces * kNormThreads * 16 * kNormRows;
      cudaError_t e = cudaFuncSetAttribute(vis_norm_sum_kernel<float>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(vis_norm_sum_kernel<__nv_bfloat16>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
      if (e != cudaSuccess) return e;
      configured[dev] = true;
    }
    const size_t smem = norm_sum_smem(a.D, a.dtype == 0 ? 4 : 2);
    dim3 gn(n_split, a.B);
    if (a.dtype == 0)
      vis_norm_sum_kernel<float><<<gn, kNormThreads, smem, s>>>(a, inv_v, ws_sum, chunk);
    else
      vis_norm_sum_kernel<__nv_bfloat16><<<gn, kNormThreads, smem, s>>>(a, inv_v, ws_sum, chunk);
  } else {
    cudaError_t e = vis_inv_norm_launch(a, inv_v, s);
    if (e != cudaSuccess) return e;
  }
  if (a.dtype == 0) {
    if (!fused) vis_sum_kernel<float><<<g1, 256, 0, s>>>(a, inv_v, ws_sum, chunk);
    vis_sum_reduce_kernel<<<g4, 256, 0, s>>>(a, ws_sum, n_split, total);
    text_mu_kernel<float><<<g2, 256, 0, s>>>(a, total, ws_mu, ws_invt);
    if (mask_ready != nullptr) {
      const cudaError_t e = cudaStreamWaitEvent(s, mask_ready, 0);  // the first kernel that reads the mask
      if (e != cudaSuccess) return e;
    }
    static std::atomic<bool> set[64];  // per device, zero-initialised
    return split::launch(relevance_kernel<float>, split::kSmem<float>, set, g3, C, s, a, C, mask, (const float*)inv_v, (const float*)ws_mu,
                         (const float*)ws_invt, p);
  } else {
    if (!fused) vis_sum_kernel<__nv_bfloat16><<<g1, 256, 0, s>>>(a, inv_v, ws_sum, chunk);
    vis_sum_reduce_kernel<<<g4, 256, 0, s>>>(a, ws_sum, n_split, total);
    text_mu_kernel<__nv_bfloat16><<<g2, 256, 0, s>>>(a, total, ws_mu, ws_invt);
    if (mask_ready != nullptr) {
      const cudaError_t e = cudaStreamWaitEvent(s, mask_ready, 0);
      if (e != cudaSuccess) return e;
    }
    static std::atomic<bool> set[64];  // per device, zero-initialised
    return split::launch(relevance_kernel<__nv_bfloat16>, split::kSmem<__nv_bfloat16>, set, g3, C, s, a, C, mask, (const float*)inv_v,
                         (const float*)ws_mu, (const float*)ws_invt, p);
  }
}

cudaError_t merge_launch(const SimArgs& a, const int* keep_idx, int keep, const float* inv_v,
                         int* assign, void* merged, float* ws_best, int* ws_bidx, int* ws_pruned,
                         void* ws_perm, int num_sms, cudaStream_t s, bool index_ready) {
  // kpos lives in `assign` until the final assignment overwrites it: it is
  // read by merge_assign_kernel (same index only).
  int* kpos = assign;
  const size_t nb = (size_t)a.B * a.N_v;
  const int tc_split = merge_tc_split(a.B, a.N_v, keep, num_sms);
  const bool tc = ws_perm != nullptr && merge_tc_supported(a, keep, tc_split);
  const int n_pruned = a.N_v - keep;
  int n_split = 1;
  // the kept-position map and the pruned rows: the FFMA Gram takes every row that is not
  // kept (clusters past the last one leave at once), the tensor-core one as many as a valid
  // keep_idx leaves
  const int cap = tc || index_ready ? n_pruned : a.N_v;
  if (!index_ready) merge_index_kernel<<<a.B, 1024, 0, s>>>(keep_idx, keep, a.N_v, kpos, ws_pruned, cap, a.err);
  if (tc) {
    cudaError_t e = merge_argmax_tc_launch(a, keep_idx, keep, inv_v, ws_pruned, ws_perm, tc_split, ws_best,
                                           ws_bidx, num_sms, &n_split, s);
    if (e != cudaSuccess) return e;
  } else if (cap > 0) {
    // column splits until three CTAs per SM are there, then the K split
    const int rt = std::max(1, (n_pruned + split::kTile - 1) / split::kTile), ct = (keep + split::kTile - 1) / split::kTile;
    n_split = (int)std::min<long long>(std::min(ct, kMergeMaxSplit), 3ll * num_sms / ((long long)rt * a.B));
    if (n_split < 1) n_split = 1;
    const int C = split::cluster_size((long long)rt * a.B * n_split, a.D, num_sms);
    const dim3 g((unsigned)(C * ((cap + split::kTile - 1) / split::kTile)), (unsigned)a.B, (unsigned)n_split);
    static std::atomic<bool> set_f32[64], set_bf16[64];  // per device, zero-initialised
    const cudaError_t e =
        a.dtype == 0 ? split::launch(merge_argmax_kernel<float>, split::kSmem<float>, set_f32, g, C, s, a, C, (const int*)ws_pruned, cap,
                                     keep_idx, keep, inv_v, n_split, ws_best, ws_bidx)
                     : split::launch(merge_argmax_kernel<__nv_bfloat16>, split::kSmem<__nv_bfloat16>, set_bf16, g, C, s, a, C, (const int*)ws_pruned,
                                     cap, keep_idx, keep, inv_v, n_split, ws_best, ws_bidx);
    if (e != cudaSuccess) return e;
  }
  // the counter of the long centroids is the last entry of the pruned list's room: past the
  // list (keep >= 1), or in it where that is full length, whose reader is done by then
  int* n_long = merged != nullptr ? ws_pruned + nb - 1 : nullptr;
  cudaError_t el = launch_pdl(merge_assign_kernel, dim3((unsigned)((nb + 255) / 256)), dim3(256), 0, s, a,
                              (const int*)kpos, n_split, (const float*)ws_best, (const int*)ws_bidx, assign,
                              n_long);
  if (el != cudaSuccess) return el;
  if (merged != nullptr) {
    // counting sort of the rows by centroid; the scratch reuses ws_best/ws_bidx
    // (the argmax partials are consumed by merge_assign_kernel above)
    int* cnt = ws_bidx;
    int* off = cnt + (size_t)a.B * keep;
    int* cur = off + (size_t)a.B * keep;
    int* lng = cur + (size_t)a.B * keep;
    int* mem = reinterpret_cast<int*>(ws_best);
    cudaError_t es = keep <= kSortSmemKeep
                         ? launch_pdl(merge_sort_kernel<true>, dim3(a.B), dim3(1024),
                                      (size_t)2 * keep * sizeof(int), s, (const int*)assign, a.N_v, keep, cnt,
                                      off, cur, mem, n_long, lng)
                         : launch_pdl(merge_sort_kernel<false>, dim3(a.B), dim3(1024), 0, s, (const int*)assign,
                                      a.N_v, keep, cnt, off, cur, mem, n_long, lng);
    if (es != cudaSuccess) return es;
    const int vec = a.dtype == 0 ? 4 : 8, n_slices = (a.D / vec + kMeanThreads - 1) / kMeanThreads;
    const int group_tasks = a.B * ((keep + kMeanGroup - 1) / kMeanGroup) * n_slices;
    // CTAs for the long centroids, which leave at once where none is long: one where
    // so few rows are pruned that none can be with a valid keep_idx, else two per SM,
    // and four beside 16 or more groups per SM, which cover the idle ones: a pass with many
    // long centroids took 179 us against 202 at 25 groups per SM and 150 against 152 at 23;
    // from 8 to 19 the two are within 1%.
    const int n_lc = n_pruned < kMeanShort ? 1 : (group_tasks >= 16 * num_sms ? 4 : 2) * num_sms;
    const dim3 gm((unsigned)(group_tasks + n_lc));
    auto go = [&](auto kernel) {
      return launch_pdl(kernel, gm, dim3(kMeanThreads), kMeanSmem, s, a, (const int*)cnt, (const int*)off,
                        (const int*)mem, keep, merged, (const int*)n_long, (const int*)lng, n_lc);
    };
    const cudaError_t em = a.dtype == 0 ? go(merge_mean_kernel<float, Sum3>)
                                        : go(merge_mean_kernel<__nv_bfloat16, float>);
    if (em != cudaSuccess) return em;
  }
  return cudaGetLastError();
}

}  // namespace provip
