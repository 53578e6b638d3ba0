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

// One k-block of a weight gradient: both operands MN-major (K runs over the expert's rows).
__device__ __forceinline__ void mma_kblock_wgrad(uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr, bool first_kblock,
                                                 int k16_steps) {
  constexpr uint32_t idesc = make_idesc_bf16(2 * BLOCK_M, BN, 1, 1);
#pragma unroll
  for (int k16 = 0; k16 < BK / 16; ++k16) {
    const uint64_t da = make_smem_desc(a_addr + k16 * 2048, MN_BOX_BYTES, 1024);
    const uint64_t db = make_smem_desc(b_addr + k16 * 2048, MN_BOX_BYTES, 1024);
    // the last k-block may hold fewer than 64 rows of the expert: the 16-row
    // steps that would only multiply zero padding are not issued
    if (k16 < k16_steps) tc_mma_bf16_pair(d_tmem, da, db, idesc, !(first_kblock && k16 == 0));
  }
}

}  // namespace moe
