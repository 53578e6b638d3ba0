// Tile-level pieces of the weight gradients on CTA pairs (tcgen05 cta_group::2): each CTA of a pair loads its
// own 128 rows of A and its half of the B tile; the even CTA issues 256 x 256 MMAs.
#pragma once

#include "gemm_tile.cuh"

namespace moe {

constexpr int HALF_B_BYTES = B_STAGE_BYTES / 2;                 // 16 KB: this CTA's half of the B tile

// 16-row MMA steps needed in k-block kb of a reduction over `rows` rows
__device__ __forceinline__ int k16_steps_of(int rows, int kb) {
  const int left = rows - kb * BK;
  return left >= BK ? BK / 16 : (left + 15) / 16;
}

}  // namespace moe
