// Tile-level building blocks of the grouped GEMMs on the sm_100a tensor cores: tile geometry and staging.
//
// Tiles never straddle experts: rows live in a padded row space where every expert segment starts
// on a multiple of 128 (the paper's rule that vector tiles align with GMM row partitions and that
// the reduction dimension stays intact, Section 4.2).
#pragma once

#include "moe_internal.h"

namespace moe {

constexpr int BN = 256;                       // accumulator columns per tile
constexpr int BK = 64;                        // reduction elements per stage (one 128-byte swizzle row)
constexpr int A_STAGE_BYTES = BLOCK_M * BK * 2;  // 16 KB
constexpr int B_STAGE_BYTES = BN * BK * 2;       // 32 KB
constexpr int MN_BOX_BYTES = 64 * BK * 2;        // one [64 k][64 mn] box of an MN-major operand
constexpr int HALF_B_BYTES = B_STAGE_BYTES / 2;  // 16 KB: a CTA's half of a pair's B tile
constexpr int TMEM_COLS = 512;
constexpr int OUT_BOX_BYTES = 32 * 64 * 2;       // epilogue staging box: 32 rows x 64 bf16 columns

struct Tile {   // of a weight gradient
  int e;      // expert
  int n0;     // first output column of the tile
  int m0;     // first output row (within the expert's slab)
  int nkb;    // k-blocks of the main loop (0 for an expert without rows)
};

// 16-row MMA steps needed in k-block kb of a reduction over `rows` rows
__device__ __forceinline__ int k16_steps_of(int rows, int kb) {
  const int left = rows - kb * BK;
  return left >= BK ? BK / 16 : (left + 15) / 16;
}

// ---------------------------------------------------------------- epilogues
// Weight gradients: an epilogue warp owns 32 rows of the tile (its TMEM lane quadrant) and private staging boxes of
// [32 rows][64 columns] bf16 in the 128-byte-swizzled layout the store tensor maps expect.
// A thread (= one row) writes 16-byte chunks at chunk index (j ^ (row & 7)): conflict-free.
__device__ __forceinline__ void stage8(uint8_t* box, int lane, int j, const float* v) {
  uint4 q = make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                       pack_bf16x2(v[6], v[7]));
  *reinterpret_cast<uint4*>(box + lane * 128 + ((j ^ (lane & 7)) << 4)) = q;
}

// After filling: publish the writes to the async proxy; lane 0 then issues the stores.
__device__ __forceinline__ void staging_release() {
  fence_proxy_async_smem();
  __syncwarp();
}

}  // namespace moe
