// CUDA-core (FFMA) "NT" products C = A * B^T over long rows (the pre-LLM pass's
// K is the embedding width, thousands of elements, while its tiles are few): a
// 64 x 64 tile per cluster of CTAs, each CTA taking a contiguous share of K, the
// shares added in order over distributed shared memory.
//
// A 256-thread CTA computes a 64 x 64 tile of its share. Steps of 32 elements of
// every row arrive in a ring of four (cp.async, three steps ahead: a step's FMAs
// take about 0.5 us alone on an SM, a load from HBM more than 1). Each half of the
// CTA multiplies half of a step (two warps per scheduler: one alone waits for
// its own shared-memory reads), and the halves are added at the end. Thread
// (rg = tid / 16 % 8, kg = tid % 16) of a half owns rows rg + 8 i (i < 8) and
// columns kg + 16 j (j < 4). A 128 x 64 tile without the split or
// the ring took 2.4 us per step and had all of K to itself:
// 311 us for the Gram of 64 text rows of 4096 elements, 367 for their products
// with 576 visual rows, 411 for 384 pruned by 192 kept rows, on 1, 9 and 15 CTAs;
// this form takes 21 (8 CTAs; the Gram now takes two parts of 8), 25 and 37 (72 and 144
// CTAs), about 42% of the issue slots between the ring's start and the last step. The shorter sums are closer to 64
// bits: p to 1.2e-7 where it was 1.1e-6.
#pragma once

#include "common.cuh"

namespace provip {
namespace split {

constexpr int kTile = 64;
constexpr int kThreads = 256;
constexpr int kKT = 32;
constexpr int kStages = 4;
constexpr int kPartLD = kTile + 4;  // padded row of a tile part (floats)
constexpr int kMaxCluster = 8;
constexpr int kCtasPerSm = 2;
// a row of a step in shared memory, padded so that 16 rows' 16-byte pieces meet
// every bank the fewest times
template <typename T>
constexpr int kPitch = kKT * (int)sizeof(T) + 16;
template <typename T>
constexpr size_t kSmem = (size_t)kStages * 2 * kTile * kPitch<T>;
static_assert(kSmem<__nv_bfloat16> >= kTile * kPartLD * sizeof(float), "the tile part takes the ring's place");

// four consecutive elements of a row in shared memory
__device__ __forceinline__ float4 frag4(const uint8_t* p, const float*) {
  return *reinterpret_cast<const float4*>(p);
}
__device__ __forceinline__ float4 frag4(const uint8_t* p, const __nv_bfloat16*) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// this CTA's share [k0, k1) of kdim elements (multiples of 8) among C
__device__ __forceinline__ void share(int kdim, int rank, int C, int& k0, int& k1) {
  const int n8 = kdim / 8;
  k0 = (int)((long long)n8 * rank / C) * 8;
  k1 = (int)((long long)n8 * (rank + 1) / C) * 8;
}

// part[64][kPartLD] (at the start of the ring) = the tile's products over elements
// [k0, k1) of the rows (null: a zero row). Every thread of the block takes part;
// ends with a block barrier. any: a valid address, never read through.
template <typename T>
__device__ __forceinline__ void tile_part(const T* const* arow, const T* const* brow, int k0, int k1,
                                          uint8_t* ring, const void* any) {
  constexpr int kVec = 16 / (int)sizeof(T);  // elements per 16-byte copy
  constexpr int kPer = kKT / kVec;           // copies per row of a step
  const int tid = threadIdx.x, half = tid >> 7, rg = (tid >> 4) & 7, kg = tid & 15;
  // thread t copies piece t % kPer of rows t / kPer, + 256 / kPer, .. (A then B)
  constexpr int kCopies = 2 * kTile * kPer / kThreads;
  const int lc = (tid % kPer) * kVec;
  const int n = k1 > k0 ? (k1 - k0 + kKT - 1) / kKT : 0;
  // one group per step, empty past the last, so that a fixed count is in flight
  auto fetch = [&](int i) {
    if (i < n) {
      const int k = k0 + i * kKT + lc;
      uint8_t* dst = ring + (size_t)(i % kStages) * 2 * kTile * kPitch<T> + (size_t)(tid / kPer) * kPitch<T> +
                     (tid % kPer) * 16;
#pragma unroll
      for (int q = 0; q < kCopies; ++q) {
        const int r = tid / kPer + q * (kThreads / kPer);
        const T* src = r < kTile ? arow[r] : brow[r - kTile];
        const bool ok = src != nullptr && k < k1;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                         smem_u32(dst + (size_t)q * (kThreads / kPer) * kPitch<T>)),
                     "l"(ok ? src + k : static_cast<const T*>(any)), "r"(ok ? 16 : 0)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll 1
  for (int i = 0; i < kStages - 1; ++i) fetch(i);
#pragma unroll 1
  for (int st = 0; st < n; ++st) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();  // step st is there for every thread, and step st - 1 has been read
    fetch(st + kStages - 1);
    const uint8_t* A = ring + (size_t)(st % kStages) * 2 * kTile * kPitch<T>;
    const uint8_t* B = A + (size_t)kTile * kPitch<T>;
#pragma unroll
    for (int kq = 0; kq < kKT / 2; kq += 4) {
      const int kk = half * (kKT / 2) + kq;
      float4 a[8], b[4];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        a[i] = frag4(A + (size_t)(rg + 8 * i) * kPitch<T> + kk * sizeof(T), static_cast<const T*>(nullptr));
#pragma unroll
      for (int j = 0; j < 4; ++j)
        b[j] = frag4(B + (size_t)(kg + 16 * j) * kPitch<T> + kk * sizeof(T), static_cast<const T*>(nullptr));
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
          acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
          acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
          acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
        }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();  // the last step has been read, and no copy is in flight
  float* part = reinterpret_cast<float*>(ring);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (half == h)
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float* o = part + (rg + 8 * i) * kPartLD + kg + 16 * j;
          *o = h == 0 ? acc[i][j] : *o + acc[i][j];
        }
    __syncthreads();
  }
}

// columns [c, c + 4) of row r of the tile: the C parts added in order (after a
// cluster barrier)
__device__ __forceinline__ float4 sum_parts(const uint8_t* ring, int r, int c, int C) {
  const uint32_t local = smem_u32(ring) + (uint32_t)(r * kPartLD + c) * (uint32_t)sizeof(float);
  float4 v[kMaxCluster];
#pragma unroll
  for (int q = 0; q < kMaxCluster; ++q)
    if (q < C) {
      uint32_t addr;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(local), "r"(q));
      asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
                   : "=f"(v[q].x), "=f"(v[q].y), "=f"(v[q].z), "=f"(v[q].w)
                   : "r"(addr)
                   : "memory");
    }
  float4 s = v[0];
#pragma unroll
  for (int q = 1; q < kMaxCluster; ++q)
    if (q < C) {
      s.x += v[q].x;
      s.y += v[q].y;
      s.z += v[q].z;
      s.w += v[q].w;
    }
  return s;
}

// reductions across the 16 lanes that share a row of a tile
__device__ __forceinline__ float row16_max(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float row16_sum(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// CTAs per cluster for `tiles` clusters over kdim elements: the most that keep
// the grid within the CTAs that are resident at once and a share of at least four
// K steps
inline int cluster_size(long long tiles, int kdim, int num_sms) {
  int C = kMaxCluster;
  while (C > 1 && (tiles * C > (long long)kCtasPerSm * num_sms || kdim / C < 4 * kKT)) C /= 2;
  return C;
}

// smem: kSmem<T> of the kernel's rows; set: its per-device flags
template <typename... P, typename... A>
inline cudaError_t launch(void (*k)(P...), size_t smem, std::atomic<bool>* set, dim3 grid, int C, cudaStream_t s,
                          A&&... args) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !set[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    set[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, static_cast<A&&>(args)...);
}

}  // namespace split
}  // namespace provip
