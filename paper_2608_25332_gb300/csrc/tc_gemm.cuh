// Tile sizes shared by the warp-specialised tcgen05 Grams of the pre-LLM pass
// (Sec. 4.2-4.3): 128 rows by 64-element K slices (128-byte swizzled TMA rows),
// warp 0 loading, warp 1 issuing the MMAs, the other warps reading the
// accumulators. Every mbarrier wait is bounded (mbar_wait); a timeout marks the
// CTA failed, and the roles drain and exit.
#pragma once

#include "common.cuh"

namespace provip {
namespace tcg {

constexpr int kBM = 128;
constexpr int kBK = 64;                      // bf16 elements per stage row (128 B)
constexpr int kABytes = kBM * kBK * 2;       // 16 KiB
constexpr int kThreads = 192;                // 6 warps

}  // namespace tcg
}  // namespace provip
