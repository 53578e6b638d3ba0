// Token-column tiles of the row-space grouped GEMMs (GMM1+SwiGLU, GMM2, act_grad, gate_grad) on CTA
// pairs.  The weights take the 256 accumulator ROWS of a pair (128 per CTA, the A operand of
// tcgen05.mma) and the expert's tokens the accumulator COLUMNS (the B operand, 32..256 per tile in
// steps of 32, half of them in each CTA's shared memory).  The MMA time of a tile then follows the
// number of tokens it really holds instead of the padded 256 rows of a token-row tile.
//
// The accumulator arrives transposed (TMEM lane = output feature, column = token); the epilogues write it back token-major:
// transposing stmatrix into a small staging box of the warp's own, read back by rows, plain 16-byte stores.
#pragma once

#include <cuda_bf16.h>

#include "gemm_tile.cuh"

namespace moe {

constexpr int TOK_GRAIN = 32;                    // tokens per tile: a multiple of 32 (16 rows of B per CTA)
constexpr int W_STAGE_BYTES = A_STAGE_BYTES;     // 128 weight rows (or 2 MN-major boxes) x 64 k: 16 KB

struct SwapTile {
  int row0;   // first padded row of the tile's tokens, a multiple of BLOCK_M
  int ntok;   // tokens (accumulator columns) of the tile, multiple of TOK_GRAIN
  int n0;     // first output feature of the pair (GATE_UP: of the 128 gate/up feature pairs)
  int nb;     // feature-tile index
};
// M-blocks of `rows` consecutive rows from the first row of an M-block on (their event counters)
__device__ __forceinline__ int mblocks_of(int rows) { return (rows + BLOCK_M - 1) / BLOCK_M; }

// Features per pair tile: GATE_UP holds 64 gate + 64 up rows per CTA = 128 features per pair.
template <int MODE>
__device__ __forceinline__ int swap_tile_features() { return MODE == GEMM_GATE_UP ? 128 : 256; }

// Tokens of the unit of M-blocks [first, first + count) (relative to the expert's first M-block) of an expert of `rows` rows,
// cut at the expert's last 32-row group.
__device__ __forceinline__ int unit_tokens(int rows, int first, int count) {
  return min((first + count) * BLOCK_M, (rows + TOK_GRAIN - 1) & ~(TOK_GRAIN - 1)) - first * BLOCK_M;
}

// One work item of a row-space operator: a token tile, or -- for an expert that merges (schedule.h) -- its last two token
// tiles (one block; block + tail) under ONE k-loop: the weight stage is written to shared memory once and multiplied with
// both token tiles into two accumulators (shared-memory traffic bounds these kernels, and the
// weights are the larger half of it).  For the epilogue warps the item is two tiles.
struct SwapWork {
  int e, n0, nb, nkb;   // expert, tile of features as in SwapTile, k-blocks
  int row0;             // first padded row
  int ntok, ntok_b;     // tokens of the tile; of the second one, whose rows follow (then ntok is BLOCK_M), 0 if the item is one tile
};
__device__ __forceinline__ int total_swap_work(const GemmArgs& a) { return a.meta[4] * a.n_tiles_n; }

// Item order: expert-major; inside an expert the feature tile is the slow index and the item the
// fast one (items running at the same time share one slab of weights in L2).
template <int MODE>
__device__ __forceinline__ SwapWork decode_swap_work(const GemmArgs& a, int t) {
  const SwapItem it = decode_swap_item(t, a.n_tiles_n, a.work_start, a.wblk_expert, a.mb_start);
  SwapWork w;
  w.e = it.e;
  w.nb = it.nb;
  w.n0 = it.nb * swap_tile_features<MODE>();
  w.nkb = (a.K + BK - 1) / BK;
  w.row0 = it.mb_first * BLOCK_M;
  const int rel = it.mb_first - a.mb_start[it.e], rows = a.counts[it.e];
  w.ntok = unit_tokens(rows, rel, it.mb_count_a);
  w.ntok_b = it.merged ? unit_tokens(rows, rel + it.mb_count_a, it.mb_count - it.mb_count_a) : 0;
  return w;
}

__device__ __forceinline__ uint32_t swap_stage_tx_bytes(int ntok) {
  return 2u * (uint32_t)(W_STAGE_BYTES + (ntok >> 1) * BK * 2);   // both CTAs: weights + half of the tokens
}

// This CTA's loads of one k-block are split over two producer warps.  Tokens: rows [row0 + rank * ntok/2, + ntok/2) as ONE
// box (a tensor map per box height).  The even CTA's weight producer arms the barrier for both CTAs' bytes.
__device__ __forceinline__ void load_tokens_swap(const GemmArgs& a, int row0, int half, int kb, int rank, uint8_t* sT,
                                                 uint64_t* bar) {
  // half: a multiple of 16, at most 128: one box of exactly that many rows
  tma_load_2d_pair(sT, &a.tmTok[(half >> 4) - 1], kb * BK, row0 + rank * half, bar);
}
__device__ __forceinline__ void load_weights_swap(GemmMode mode, const GemmArgs& a, int e, int n0, int kb, int rank, uint8_t* sW,
                                                  uint64_t* bar, int ntok_total) {
  const int k0 = kb * BK;
  if (rank == 0) mbar_expect_tx_elect(bar, swap_stage_tx_bytes(ntok_total));
  const int brow = e * a.b_rows_per_expert;
  if (mode == GEMM_GATE_UP) {
    // one box [8 groups][gate | up][8 rows][64 k]: per group of 8 features the 8 gate rows, then the 8 up rows
    // (W_gate_up viewed as [Ep][F/8][2][8][d]); groups beyond F read as zeros
    tma_load_5d_pair(sW, &a.tmB, k0, 0, 0, (n0 + rank * 64) >> 3, e, bar);
  } else if (mode == GEMM_DOWN) {
    tma_load_2d_pair(sW, &a.tmB, k0, brow + n0 + rank * 128, bar);
  } else {
    // ACT_GRAD / GATE_GRAD: the forward weight read along its rows -> two MN-major [64 k][64 features] boxes
    tma_load_2d_pair(sW, &a.tmB, n0 + 2 * rank * 64, brow + k0, bar);
    tma_load_2d_pair(sW + MN_BOX_BYTES, &a.tmB, n0 + (2 * rank + 1) * 64, brow + k0, bar);
  }
}

// One 64-deep k-block: D[256 features x ntok tokens] (+)= W . X^T.  w_lo / t_lo: low descriptor words of
// the stage's weight and token tiles (smem_desc_lo).
template <bool W_MN>   // act_grad, gate_grad: the forward weights read along their rows
__device__ __forceinline__ void mma_kblock_swap(uint32_t d_tmem, uint32_t w_lo, uint32_t t_lo, uint32_t idesc,
                                                bool first_kblock) {
  // 16 k-rows of an MN-major box / 32 bytes of a K-major row
  tc_mma4_bf16_pair<W_MN ? (2048 >> 4) : (32 >> 4), (32 >> 4)>(d_tmem, w_lo, t_lo, smem_desc_hi(1024), idesc, !first_kblock);
}
template <bool W_MN>
__device__ __forceinline__ uint32_t swap_w_desc_lo(uint32_t w_addr) {
  return smem_desc_lo(w_addr, W_MN ? MN_BOX_BYTES : 16);
}
template <bool W_MN>
__device__ __forceinline__ uint32_t swap_idesc(int ntok) {
  return make_idesc_bf16(2 * BLOCK_M, ntok, W_MN ? 1 : 0, 0);
}

// ---------------------------------------------------------------- staging of an epilogue warp
// A warp takes a chunk of tokens from TMEM as matrix fragments (pairs of tokens of one feature per register pair), writes
// the bf16 results to its staging with transposing stmatrix -- rows of tokens there -- reads them back by row and stores
// 16-byte vectors.  Nothing but the warp itself waits for the staging.  Rows of 32 or 64 bytes; their 16-byte
// pieces are permuted so that the eight rows of a matrix fall into different banks.
template <int MODE>
__host__ __device__ constexpr int sw_chunk() { return MODE == GEMM_ACT_GRAD ? 16 : 32; }   // tokens of a chunk
// Staging bytes of a warp.  gate+up: [32 tokens][16 features] of A, H gate, H up (down: the same, one layout in the persistent
// forward launch); act_grad: [gate | up][16 tokens][32 features], the pre-activations in, their gradients out; gate_grad, down:
// [32 tokens][32 features].
__host__ __device__ constexpr int sw_staging_bytes(GemmMode mode) { return mode == GEMM_ACT_GRAD || mode == GEMM_GATE_GRAD ? 2048 : 3072; }
// byte offset of 16-byte piece c of token t in rows of 64 and of 32 bytes
__device__ __forceinline__ uint32_t piece64(int t, int c) { return t * 64 + ((c ^ ((t >> 1) & 3)) << 4); }
__device__ __forceinline__ uint32_t piece32(int t, int c) { return t * 32 + ((c ^ ((t >> 2) & 1)) << 4); }
__device__ __forceinline__ uint4 ld_nc_v4(const uint16_t* p) {
  uint4 r;
  asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}


// 1 / (1 + e^-g) of two values
__device__ __forceinline__ float2x sigmoid2(float2x g) {
  float lo, hi;
  unpack2(mul2(g, pack2(-1.4426950408889634f, -1.4426950408889634f)), lo, hi);
  asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(lo));
  asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(hi));
  unpack2(add2(pack2(lo, hi), pack2(1.0f, 1.0f)), lo, hi);
  asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(lo));
  asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(hi));
  return pack2(lo, hi);
}

// ---------------------------------------------------------------- epilogues (transposed accumulator)
// Warps `quad` and `quad + 4` of CTA `rank` own TMEM lanes 32*quad .. 32*quad+31 (32 output features) and walk the tile's
// tokens in alternating chunks: latency, two warps hide each other's.  `ready` waits for the accumulator; what a chunk needs
// besides it is fetched before.
//
// What bounds it is instructions: with a feature per lane, 2-byte staging accesses and shuffles between gate and up lanes
// act_grad took 675 instructions per 16 tokens and warp, 19 us for a 256-token tile (gate+up with H kept 12 us, down 6 us) -- on
// passes with a few tiles per SM longer than their MMAs, and exposed.
template <int MODE, class READY>
__device__ __forceinline__ bool epilogue_swap(const GemmArgs& a, const SwapTile& st, uint32_t tmem_acc, int rank,
                                              int ew, int lane, uint8_t* staging, READY ready) {
  const int quad = ew & 3;
  constexpr int CH = sw_chunk<MODE>();
  const int first = (ew >> 2) * CH;
  const uint32_t trow = tmem_acc + (static_cast<uint32_t>(quad * 32) << 16);
  constexpr uint32_t HALF = 16u << 16;   // TMEM lanes 16.. of the warp
  const uint32_t stg = smem_u32(staging);
  const int mrow = lane & 7, mat = lane >> 3;   // this lane gives the address of row mrow of matrix mat
  if (MODE == GEMM_DOWN || MODE == GEMM_GATE_GRAD) {
    if (!ready()) return false;
    const int f0 = st.n0 + rank * 128 + quad * 32;   // first output column of this warp
    if (f0 >= a.N) return true;
    const int part = lane & 3;
    const bool inside = f0 + part * 8 < a.N;     // N % 8 == 0: a 16-byte piece is inside or outside as a whole
    const size_t ld = row_ld(a.N);
    uint16_t* const out = a.out0 + st.row0 * ld + f0 + part * 8;
#pragma unroll 1
    for (int c0 = first; c0 < st.ntok; c0 += 2 * CH) {
      float v[32];   // [features 0.. | 16..][token group of 8][feature, feature + 8][token pair]
      tmem_ld_frag4(trow + c0, v);
      tmem_ld_frag4(trow + HALF + c0, v + 16);
      tmem_ld_wait();
      __syncwarp();   // the chunk before has been read back
#pragma unroll
      for (int f = 0; f < 4; ++f) {   // 8 features: matrices of the four token groups
        const float* p = v + 16 * (f >> 1) + 2 * (f & 1);
        stmatrix4_trans(stg + piece64(8 * mat + mrow, f), pack_bf16x2(p[0], p[1]), pack_bf16x2(p[4], p[5]),
                        pack_bf16x2(p[8], p[9]), pack_bf16x2(p[12], p[13]));
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int t = (lane + 32 * i) >> 2;
        const uint4 q = *reinterpret_cast<const uint4*>(staging + piece64(t, part));
        if (inside) *reinterpret_cast<uint4*>(out + (c0 + t) * ld) = q;
      }
    }
  } else if (MODE == GEMM_GATE_UP) {
    // TMEM lanes 0..7 and 16..23: gate pre-activations of features 0..7 and 8..15 of the warp, lanes 8..15 and 24..31: up
    // pre-activations of the same features: a fragment holds both of a feature in one thread.
    const int fw0 = st.n0 + rank * 64 + quad * 16;   // first feature of this warp
    const float* wsrc = a.prow_w + st.row0 + 2 * (lane & 3);   // routing weights of the thread's token pairs
    float2 w_next[4];
    auto fetch = [&](int c0) {
#pragma unroll
      for (int b = 0; b < 4; ++b) w_next[b] = *reinterpret_cast<const float2*>(wsrc + c0 + 8 * b);
    };
    if (!ready()) return false;   // (the weights are complete with the tokens, which the MMAs have read)
    if (fw0 >= a.F) return true;
    if (first < st.ntok) fetch(first);
    const int part = lane & 1;
    const bool inside = fw0 + 8 * part < a.F;     // F % 8 == 0
    const size_t col = fw0 + 8 * part, ld_a = row_ld(a.F), ld_h = row_ld(2 * a.F);
#pragma unroll 1
    for (int c0 = first; c0 < st.ntok; c0 += 2 * CH) {
      float v[32];   // [features 0..7 | 8..15][token group of 8][gate, up][token pair]
      tmem_ld_frag4(trow + c0, v);
      tmem_ld_frag4(trow + HALF + c0, v + 16);
      float2x w[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) w[b] = pack2(w_next[b].x, w_next[b].y);
      if (c0 + 2 * CH < st.ntok) fetch(c0 + 2 * CH);
      tmem_ld_wait();
      __syncwarp();   // the chunk before has been read back
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t act[4], hg[4], hu[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const float* p = v + 16 * h + 4 * b;
          const float2x g = pack2(p[0], p[1]), u = pack2(p[2], p[3]);
          act[b] = pack_bf16x2(mul2(w[b], mul2(mul2(g, sigmoid2(g)), u)));
          hg[b] = pack_bf16x2(p[0], p[1]);
          hu[b] = pack_bf16x2(p[2], p[3]);
        }
        const uint32_t at = stg + piece32(8 * mat + mrow, h);
        stmatrix4_trans(at, act[0], act[1], act[2], act[3]);
        if (a.out1) {
          stmatrix4_trans(at + 1024, hg[0], hg[1], hg[2], hg[3]);
          stmatrix4_trans(at + 2048, hu[0], hu[1], hu[2], hu[3]);
        }
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int t = (lane + 32 * i) >> 1;
        const uint8_t* piece = staging + piece32(t, part);
        const size_t row = st.row0 + c0 + t;
        if (inside) {
          *reinterpret_cast<uint4*>(a.out0 + row * ld_a + col) = *reinterpret_cast<const uint4*>(piece);
          if (a.out1) {
            *reinterpret_cast<uint4*>(a.out1 + row * ld_h + col) = *reinterpret_cast<const uint4*>(piece + 1024);
            *reinterpret_cast<uint4*>(a.out1 + row * ld_h + a.F + col) = *reinterpret_cast<const uint4*>(piece + 2048);
          }
        }
      }
    }
  } else if (MODE == GEMM_ACT_GRAD) {
    const int f0 = st.n0 + rank * 128 + quad * 32;
    const int nparts = a.n_tiles_n * DW_PARTS_PER_TILE;
    const int slot = (st.nb * 2 + rank) * 4 + quad;
    if (f0 >= a.F) {
      // no features here: the partial slots of this warp still take part in the reduction
      if (!ready()) return false;
      if (a.dw_partial)
        for (int j = lane + 32 * (ew >> 2); j < st.ntok; j += 64) a.dw_partial[(size_t)(st.row0 + j) * nparts + slot] = 0.f;
      return true;
    }
    // The saved pre-activations of 16 tokens x 32 features (gate and up: 1 KB each) come in as four
    // 16-byte loads per lane (lane -> token (lane + 32 i) / 4, features 8 (lane % 4) ..), are parked in
    // this warp's staging, read as fragments, replaced there by their gradients and read back by rows.
    // The loads of the next 16 tokens are in flight while the current ones are worked on; pre-activations and routing weights
    // are the forward launch's, so the first ones are on their way before the accumulator is ready.
    const int part = lane & 3;
    const bool inside = f0 + part * 8 < a.F;     // F % 8 == 0
    const size_t ld = row_ld(2 * a.F);           // H and dH
    const uint16_t* hbase = a.in0 + st.row0 * ld + f0 + part * 8;
    uint16_t* const out = a.out0 + st.row0 * ld + f0 + part * 8;
    const float* wsrc = a.prow_w + st.row0 + 2 * (lane & 3);
    uint4 pre[4];
    float2 w_next[2];
    auto fetch = [&](int tok0) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint16_t* p = hbase + (tok0 + ((lane + 32 * i) >> 2)) * ld;
        pre[2 * i] = inside ? ld_nc_v4(p) : make_uint4(0, 0, 0, 0);
        pre[2 * i + 1] = inside ? ld_nc_v4(p + a.F) : make_uint4(0, 0, 0, 0);
        w_next[i] = *reinterpret_cast<const float2*>(wsrc + tok0 + 8 * i);
      }
    };
    if (first < st.ntok) fetch(first);
    if (!ready()) return false;
    const float2x one = pack2(1.0f, 1.0f), minus = pack2(-1.0f, -1.0f);
#pragma unroll 1
    for (int h0 = first; h0 < st.ntok; h0 += 2 * CH) {
      float da[16];   // [features 0.. | 16..][token group of 8][feature, feature + 8][token pair]
      tmem_ld_frag2(trow + h0, da);
      tmem_ld_frag2(trow + HALF + h0, da + 8);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        uint8_t* piece = staging + piece64((lane + 32 * i) >> 2, part);
        *reinterpret_cast<uint4*>(piece) = pre[2 * i];
        *reinterpret_cast<uint4*>(piece + 1024) = pre[2 * i + 1];
      }
      float2x w[2] = {pack2(w_next[0].x, w_next[0].y), pack2(w_next[1].x, w_next[1].y)};
      if (h0 + 2 * CH < st.ntok) fetch(h0 + 2 * CH);
      __syncwarp();
      tmem_ld_wait();
      float2x pr[2] = {pack2(0.f, 0.f), pack2(0.f, 0.f)};   // <dA_unweighted, a> over the thread's features, by token group
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        // matrices of (token group b, 8 features): q = 2 b + feature group
        const uint32_t at = stg + piece64(8 * (mat >> 1) + mrow, 2 * h + (mat & 1));
        uint32_t gr[4], ur[4];
        ldmatrix4_trans(at, gr);
        ldmatrix4_trans(at + 1024, ur);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int b = q >> 1;
          const float* p = da + 8 * h + 4 * b + 2 * (q & 1);
          const float2x g = pack2(bf16lo(gr[q]), bf16hi(gr[q])), u = pack2(bf16lo(ur[q]), bf16hi(ur[q])), d = pack2(p[0], p[1]);
          const float2x s = sigmoid2(g), gs = mul2(g, s);
          pr[b] = add2(pr[b], mul2(d, mul2(gs, u)));
          const float2x dav = mul2(w[b], d);          // backward Dispatch's weight, applied here
          const float2x ds = mul2(s, fma2(g, fma2(s, minus, one), one));   // derivative of g sigmoid(g)
          gr[q] = pack_bf16x2(mul2(mul2(dav, u), ds));
          ur[q] = pack_bf16x2(mul2(dav, gs));
        }
        stmatrix4_trans(at, gr[0], gr[1], gr[2], gr[3]);   // the pieces that this half's ldmatrix has read
        stmatrix4_trans(at + 1024, ur[0], ur[1], ur[2], ur[3]);
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int t = (lane + 32 * i) >> 2;
        const uint4 dg = *reinterpret_cast<const uint4*>(staging + piece64(t, part));
        const uint4 du = *reinterpret_cast<const uint4*>(staging + 1024 + piece64(t, part));
        if (inside) {
          *reinterpret_cast<uint4*>(out + (h0 + t) * ld) = dg;
          *reinterpret_cast<uint4*>(out + (h0 + t) * ld + a.F) = du;
        }
      }
      if (a.dw_partial) {
        // sum over the warp's 32 features: eight threads hold the same token pairs; each step halves what a thread keeps
        float k0, k1, s0, s1;
        const bool up = (lane & 16) != 0, odd = (lane & 8) != 0;
        unpack2(up ? pr[1] : pr[0], k0, k1);
        unpack2(up ? pr[0] : pr[1], s0, s1);
        k0 += __shfl_xor_sync(0xffffffffu, s0, 16);
        k1 += __shfl_xor_sync(0xffffffffu, s1, 16);
        float v = (odd ? k1 : k0) + __shfl_xor_sync(0xffffffffu, odd ? k0 : k1, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        const int t = (up ? 8 : 0) + 2 * (lane & 3) + (odd ? 1 : 0);
        if ((lane & 4) == 0) a.dw_partial[(size_t)(st.row0 + h0 + t) * nparts + slot] = v;
      }
      __syncwarp();   // the staging has been read back
    }
  }
  return true;
}

}  // namespace moe
