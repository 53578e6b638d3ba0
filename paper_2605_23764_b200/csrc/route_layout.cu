// Routing (softmax top-k) and the dispatch layout (per-expert histogram, prefix scan, stable
// permutation, M-block table).  Integer results are bit-exact by construction: every count and
// rank is an integer sum whose value does not depend on evaluation order.
#include <limits.h>

#include <mutex>

#include "launch_pairs.cuh"
#include "moe_internal.h"
#include "topk.cuh"

namespace moe {

// ------------------------------------------------------------------------------------------
// Router: one warp per token.  Expert e is held by lane e%32 in register e/32.
// Selection compares raw logits (softmax is monotone), ties go to the lower expert id, slots
// come out in descending logit order.  Scores: fp32 softmax over all E, max-subtracted -- or, in the
// sigmoid gate mode, 1 / (1 + exp(-logit)) per selected expert; `renorm` holds the gate mode bits.
// ------------------------------------------------------------------------------------------
template <int NPL>
__global__ void __launch_bounds__(256) route_kernel(const float* __restrict__ logits, int T, int E, int k,
                                                     int renorm, int* __restrict__ topk_ids,
                                                     float* __restrict__ topk_w, int* __restrict__ counts) {
  __shared__ uint64_t pool[8][TOPK_POOL];
  const int lane = threadIdx.x & 31;
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  pdl_wait();
  pdl_trigger();
  if (t >= T) return;
  const float* row = logits + (size_t)t * E;
  float v[NPL];
#pragma unroll
  for (int i = 0; i < NPL; ++i) {
    int e = i * 32 + lane;
    v[i] = e < E ? row[e] : -INFINITY;
  }
  uint32_t key[1][NPL];
#pragma unroll
  for (int i = 0; i < NPL; ++i) key[0][i] = i * 32 + lane < E ? float_key(v[i]) : 0u;
  int ids[1] = {0};
  float ls[1] = {0.f};
  warp_topk<NPL, 1>(key, k, lane, pool[threadIdx.x >> 5], ids, ls);
  const int my_id = ids[0];
  const float my_l = ls[0];
  float my_p;
  if (renorm & GATE_SIGMOID) {
    my_p = 1.0f / (1.0f + expf(-my_l));
  } else {
    const float mx = __shfl_sync(0xffffffffu, my_l, 0);
    float den = 0.f;
#pragma unroll
    for (int i = 0; i < NPL; ++i)
      if (i * 32 + lane < E) den += expf(v[i] - mx);
#pragma unroll
    for (int off = 16; off; off >>= 1) den += __shfl_xor_sync(0xffffffffu, den, off);
    my_p = expf(my_l - mx) / den;
  }
  if (renorm & GATE_RENORM) {
    float wsum = 0.f;
    for (int j = 0; j < k; ++j) wsum += __shfl_sync(0xffffffffu, my_p, j);
    my_p /= wsum;
  }
  if (lane < k) {
    topk_ids[(size_t)t * k + lane] = my_id;
    topk_w[(size_t)t * k + lane] = my_p;
    if (counts) atomicAdd(&counts[my_id], 1);
  }
}

cudaError_t launch_route(const float* logits, int T, int E, int k, int gate_mode, int* topk_ids, float* topk_w,
                         int* counts, cudaStream_t s, int* launches) {
  if (T == 0) return cudaSuccess;
  if (counts) {
    cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(int) * (size_t)E, s);
    if (e != cudaSuccess) return e;
  }
  const int threads = 256, tokens_per_block = threads / 32;
  dim3 grid((T + tokens_per_block - 1) / tokens_per_block);
  const int npl = (E + 31) / 32;
  cudaError_t e = cudaSuccess;
#define MOE_ROUTE_CASE(N) \
  e = launch_dependent(route_kernel<N>, grid, dim3(threads), 0, s, logits, T, E, k, gate_mode, topk_ids, topk_w, counts)
  if (npl <= 1) MOE_ROUTE_CASE(1);
  else if (npl <= 2) MOE_ROUTE_CASE(2);
  else if (npl <= 4) MOE_ROUTE_CASE(4);
  else if (npl <= 8) MOE_ROUTE_CASE(8);
  else if (npl <= 16) MOE_ROUTE_CASE(16);
  else MOE_ROUTE_CASE(32);
#undef MOE_ROUTE_CASE
  ++*launches;
  return e;
}

// ------------------------------------------------------------------------------------------
// Dispatch layout.  Flat slot i = t*kp + j; block b owns slots [b*CHUNK, (b+1)*CHUNK), warp w of
// the block owns CHUNK / warps consecutive slots of it, processed 32 at a time in slot order.
//
// Three kernels -- histograms, scans, ranks -- each bound by the latency of a few dependent accesses, not by bytes: many
// warps with two or four groups of 32 slots each, every slot's id loaded before the first is used, and each kernel
// started while the one before it runs (programmatic dependent launch).  Fewer than LAYOUT_ONE_SLOTS slots (token
// generation) take one kernel of one block instead.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ int slot_expert(const int* __restrict__ ids, int i, int k, int kp, int E) {
  int t = i / kp, j = i - t * kp;
  if (j >= k) return E + (j - k);
  int e = __ldcg(ids + (size_t)t * k + j);
  return (e >= 0 && e < E) ? e : -1;
}

// zero[0, n), n a multiple of 4, 16-byte aligned: the share of thread `first` of `threads`
__device__ __forceinline__ void clear_ints(int* zero, int n, int first, int threads) {
  for (int i = first; i < n / 4; i += threads) reinterpret_cast<int4*>(zero)[i] = make_int4(0, 0, 0, 0);
}

constexpr int HIST_THREADS = 1024;
__global__ void __launch_bounds__(HIST_THREADS) layout_hist_kernel(const int* __restrict__ ids, int n, int k, int kp, int E,
                                                                   int Ep, int* __restrict__ blk_hist, int* __restrict__ tok_last,
                                                                   int* __restrict__ zero, int nzero) {
  extern __shared__ int hist[];   // [Ep]
  for (int e = threadIdx.x; e < Ep; e += HIST_THREADS) hist[e] = 0;
  pdl_wait();      // the ids; and the previous launch on the stream may still use what is cleared here
  pdl_trigger();   // behind the wait: whoever starts from here on finds the ids complete
  __syncthreads();
  const int base = blockIdx.x * LAYOUT_CHUNK + threadIdx.x;
  int e[LAYOUT_CHUNK / HIST_THREADS];
#pragma unroll
  for (int g = 0; g < LAYOUT_CHUNK / HIST_THREADS; ++g) {
    const int i = base + g * HIST_THREADS;
    e[g] = i < n ? slot_expert(ids, i, k, kp, E) : -1;
  }
  if (tok_last)   // the tokens whose first slot lies in this block's chunk
    for (int i = base; i < min(n, (int)(blockIdx.x + 1) * LAYOUT_CHUNK); i += HIST_THREADS)
      if (i % kp == 0) tok_last[i / kp] = 0;
  clear_ints(zero, nzero, blockIdx.x * HIST_THREADS + threadIdx.x, gridDim.x * HIST_THREADS);
#pragma unroll
  for (int g = 0; g < LAYOUT_CHUNK / HIST_THREADS; ++g) {
    const uint32_t peers = __match_any_sync(0xffffffffu, e[g]);
    if (e[g] >= 0 && (threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&hist[e[g]], __popc(peers));
  }
  __syncthreads();
  for (int q = threadIdx.x; q < Ep; q += HIST_THREADS) blk_hist[(size_t)blockIdx.x * Ep + q] = hist[q];
}

// Exclusive scans over the experts of a block of 1024 threads: s_counts[Ep] -> offsets of rows, M-blocks, work items,
// 32-row groups and long experts, in shared memory (each Ep + 1 long) and in the layout's tables; the rows of the largest
// expert and the number of token tiles.
constexpr int SCAN_Q = 5;
constexpr int SCAN_ROWS = SCAN_Q + 2;   // of `totals`: by warp and behind them the block's; the last rows hold maxima and sums
struct ExpertScan { int *counts, *off, *mb, *wi, *gr, *lg; };   // shared memory
__host__ __device__ constexpr int expert_scan_ints(int Ep) { return 6 * Ep + 5; }
__device__ __forceinline__ ExpertScan expert_scan_at(int* sm, int Ep) {
  return ExpertScan{sm, sm + Ep, sm + 2 * Ep + 1, sm + 3 * Ep + 2, sm + 4 * Ep + 3, sm + 5 * Ep + 4};
}
__device__ __forceinline__ void scan_experts(int E, int Ep, const LayoutView& lv, const ExpertScan& sc, int (*totals)[33],
                                             bool write = true) {
  constexpr int NQ = SCAN_Q;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int carry[NQ] = {0, 0, 0, 0, 0}, largest = 0, tiles = 0;
  for (int e0 = 0; e0 < Ep; e0 += 1024) {
    const int e = e0 + threadIdx.x;
    const int c = e < Ep ? sc.counts[e] : 0;
    const int m = (c + BLOCK_M - 1) / BLOCK_M;
    const int pr = (m + 1) >> 1;  // token tiles (units, schedule.h)
    // work items of the token-column GEMM kernels: the units of the expert, except that an expert
    // that merges (schedule.h) has its last two units (one block; block + tail) share one k-loop
    const int val[NQ] = {c, m, pr - (expert_merges(c, m, e >= E) ? 1 : 0), (c + GROUP_ROWS - 1) / GROUP_ROWS, strip_long(c)};
    int inc[NQ] = {val[0], val[1], val[2], val[3], val[4]};
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int o = __shfl_up_sync(0xffffffffu, inc[q], off);
        if (lane >= off) inc[q] += o;
      }
    }
    if (lane == 31) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) totals[q][warp] = inc[q];
    }
    const int most = __reduce_max_sync(0xffffffffu, c), prs = __reduce_add_sync(0xffffffffu, pr);
    if (lane == 0) { totals[NQ][warp] = most; totals[NQ + 1][warp] = prs; }
    __syncthreads();
    if (warp < NQ) {   // warp q: exclusive scan of quantity q's warp totals, the block's total behind them
      const int w = totals[warp][lane];
      int wi = w;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, wi, off);
        if (lane >= off) wi += o;
      }
      totals[warp][lane] = wi - w;
      if (lane == 31) totals[warp][32] = wi;
    } else if (warp == NQ) {
      const int m = __reduce_max_sync(0xffffffffu, totals[NQ][lane]);
      if (lane == 0) totals[NQ][32] = m;
    } else if (warp == NQ + 1) {
      const int n = __reduce_add_sync(0xffffffffu, totals[NQ + 1][lane]);
      if (lane == 0) totals[NQ + 1][32] = n;
    }
    __syncthreads();
    int ex[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) ex[q] = carry[q] + totals[q][warp] + inc[q] - val[q];
    if (e < Ep) {
      sc.off[e] = ex[0]; sc.mb[e] = ex[1]; sc.wi[e] = ex[2]; sc.gr[e] = ex[3]; sc.lg[e] = ex[4];
    }
    if (write && e < Ep) {
      lv.counts[e] = c;
      lv.offsets[e] = ex[0];
      lv.mb_start[e] = ex[1];
      lv.pad_off[e] = ex[1] * BLOCK_M;
      lv.work_start[e] = ex[2];
      if (lv.group_start) {
        lv.group_start[e] = ex[3];
        for (int r = c; r < val[3] * GROUP_ROWS; ++r) lv.group_slot[ex[3] * GROUP_ROWS + r] = -1;   // padding rows of the last group
      }
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) carry[q] += totals[q][32];
    largest = max(largest, totals[NQ][32]);
    tiles += totals[NQ + 1][32];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    sc.off[Ep] = carry[0]; sc.mb[Ep] = carry[1]; sc.wi[Ep] = carry[2]; sc.gr[Ep] = carry[3]; sc.lg[Ep] = carry[4];
  }
  if (write && threadIdx.x == 0) {
    lv.offsets[Ep] = carry[0];
    lv.mb_start[Ep] = carry[1];
    lv.pad_off[Ep] = carry[1] * BLOCK_M;
    lv.work_start[Ep] = carry[2];
    lv.meta[0] = carry[1];
    lv.meta[1] = carry[1] * BLOCK_M;
    lv.meta[2] = carry[0];
    lv.meta[3] = tiles;
    lv.meta[4] = carry[2];
    lv.meta[5] = carry[3];
    lv.meta[6] = carry[4];
    lv.meta[7] = largest;
    if (lv.group_start) lv.group_start[Ep] = carry[3];
  }
  __syncthreads();
  if (write && lv.wg_order)
    for (int e = threadIdx.x; e < Ep; e += 1024)
      lv.wg_order[strip_order(e, sc.counts[e], E, Ep, sc.lg[e], sc.lg[E], sc.lg[Ep])] = e;
}
// the last expert whose start is <= i
__device__ __forceinline__ int expert_at(int Ep, const int* start, int i) {
  int lo = 0, hi = Ep - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}
// this block's share of the tables: block `part` of `parts`
__device__ __forceinline__ void expert_tables(int Ep, const LayoutView& lv, const ExpertScan& sc, int part = 0, int parts = 1) {
  const int first = part * blockDim.x + threadIdx.x, step = parts * blockDim.x;
  for (int i = first; i < sc.mb[Ep]; i += step) lv.mblk_expert[i] = expert_at(Ep, sc.mb, i);
  for (int i = first; i < sc.wi[Ep]; i += step) lv.wblk_expert[i] = expert_at(Ep, sc.wi, i);
  if (lv.group_start)
    for (int i = first; i < sc.gr[Ep]; i += step) {
      const int e = expert_at(Ep, sc.gr, i);
      lv.group_row[i] = sc.mb[e] * BLOCK_M + (i - sc.gr[e]) * GROUP_ROWS;
    }
}

// One block.  (1) per expert, exclusive scan of the block histograms over blocks: a thread per expert and range of
// blocks (as many ranges as the block has threads for), so that the reads of a row are coalesced and independent;
// (2) scans over experts; (3) M-block and work-item -> expert tables.
__global__ void __launch_bounds__(1024) layout_scan_kernel(int nblk, int E, int Ep, LayoutView lv) {
  extern __shared__ int sm[];
  __shared__ int totals[SCAN_ROWS][33];
  const ExpertScan sc = expert_scan_at(sm, Ep);
  int* part = sm + expert_scan_ints(Ep);   // [ranges][Ep]
  pdl_trigger();
  pdl_wait();
  const int ranges = Ep <= 1024 ? 1024 / Ep : 1;
  const int len = (nblk + ranges - 1) / ranges;
  for (int q = threadIdx.x; q < ranges * Ep; q += 1024) {
    const int g = q / Ep, e = q - g * Ep;
    const int b1 = min(nblk, (g + 1) * len);
    int sum = 0;
#pragma unroll 8
    for (int b = g * len; b < b1; ++b) sum += __ldcg(lv.blk_hist + (size_t)b * Ep + e);
    part[q] = sum;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < Ep; e += 1024) {
    int run = 0;
    for (int g = 0; g < ranges; ++g) { const int c = part[g * Ep + e]; part[g * Ep + e] = run; run += c; }
    sc.counts[e] = run;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < ranges * Ep; q += 1024) {
    const int g = q / Ep, e = q - g * Ep;
    const int b0 = g * len, b1 = min(nblk, b0 + len);
    int run = part[q];
    for (int b = b0; b < b1; b += 8) {   // eight reads in flight, then the running sums
      int c[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) c[u] = b + u < b1 ? __ldcg(lv.blk_hist + (size_t)(b + u) * Ep + e) : 0;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (b + u < b1) { lv.blk_hist[(size_t)(b + u) * Ep + e] = run; run += c[u]; }
    }
  }
  scan_experts(E, Ep, lv, sc, totals);
  expert_tables(Ep, lv, sc);
}

// Ranks.  WARPS warps of LAYOUT_CHUNK / WARPS slots.  The part in front of pdl_wait() -- the ids, the slots' ranks
// inside their warp and the warps' histograms -- needs nothing of the scan kernel and runs beside it (this kernel starts
// once every block of the histogram kernel is past its own wait, so the ids are complete).
template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32) layout_rank_kernel(const int* __restrict__ ids, int n, int k, int kp, int E,
                                                                 int Ep, LayoutView lv, DevStatus* status) {
  constexpr int G = LAYOUT_CHUNK / WARPS / 32;   // groups of 32 slots per warp
  extern __shared__ int sm[];
  int* base = sm;                                              // [Ep] first row of this block's rows of the expert
  int* pad = sm + Ep;                                          // [Ep] padded row - row of the expert
  int* grp = sm + 2 * Ep;                                      // [Ep] place among the groups' rows - row of the expert
  int* last = sm + 3 * Ep;                                     // [LAYOUT_CHUNK / kp + 2] key of the chunk's tokens
  const int nlast = LAYOUT_CHUNK / kp + 2;
  uint16_t* whist = reinterpret_cast<uint16_t*>(last + nlast + ((nlast + Ep) & 1));   // [WARPS][Ep + (Ep & 1)]
  const int ld = Ep + (Ep & 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_trigger();
  const int i0 = blockIdx.x * LAYOUT_CHUNK + warp * (G * 32) + lane;
  int e[G], r[G];
#pragma unroll
  for (int g = 0; g < G; ++g) e[g] = i0 + 32 * g < n ? slot_expert(ids, i0 + 32 * g, k, kp, E) : -1;
  for (int q = threadIdx.x; q < WARPS * ld / 2; q += WARPS * 32) reinterpret_cast<uint32_t*>(whist)[q] = 0;
  for (int q = threadIdx.x; q < nlast; q += WARPS * 32) last[q] = 0;
  __syncthreads();
  uint16_t* mine = whist + warp * ld;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const uint32_t peers = __match_any_sync(0xffffffffu, e[g]);
    r[g] = e[g] >= 0 ? mine[e[g]] + __popc(peers & ((1u << lane) - 1u)) : 0;
    __syncwarp();
    if (e[g] >= 0 && lane == __ffs(peers) - 1) mine[e[g]] += (uint16_t)__popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // per expert: the block's rows in front of each warp's
  for (int q = threadIdx.x; q < Ep; q += WARPS * 32) {
    int run = 0;
#pragma unroll 8
    for (int w = 0; w < WARPS; ++w) {
      const int c = whist[w * ld + q];
      whist[w * ld + q] = (uint16_t)run;
      run += c;
    }
  }
  pdl_wait();
  for (int q = threadIdx.x; q < Ep; q += WARPS * 32) {
    const int off = __ldcg(lv.offsets + q);
    base[q] = off + __ldcg(lv.blk_hist + (size_t)blockIdx.x * Ep + q);
    pad[q] = __ldcg(lv.pad_off + q) - off;
    if (lv.group_start) grp[q] = __ldcg(lv.group_start + q) * GROUP_ROWS - off;
  }
  __syncthreads();
  const int t_first = blockIdx.x * LAYOUT_CHUNK / kp;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int i = i0 + 32 * g;
    if (i >= n) continue;
    if (e[g] >= 0) {
      const int row = base[e[g]] + mine[e[g]] + r[g], prow = row + pad[e[g]];
      lv.row_of[i] = row;
      lv.prow_of[i] = prow;
      lv.src_of[row] = i;
      if (lv.group_start) lv.group_slot[row + grp[e[g]]] = i;
      // the combine order's key: the token's last ROUTED row (shared experts are taken first by the persistent launch)
      if (lv.tok_last && i % kp < k) atomicMax(&last[i / kp - t_first], prow + 1);
    } else {
      lv.row_of[i] = -1;
      lv.prow_of[i] = -1;
      note(status, /*MOE_ERR_BAD_EXPERT_ID*/ 1, i);  // the slot is dropped, the layer carries on
    }
  }
  if (!lv.tok_last) return;
  __syncthreads();
  for (int q = threadIdx.x; q < nlast; q += WARPS * 32)   // a token whose slots straddle two chunks gets both chunks' keys
    if (last[q]) atomicMax(&lv.tok_last[t_first + q], last[q]);
}

// Exclusive scan of bins[nb] in shared memory by a block of 1024 threads.
__device__ __forceinline__ void scan_bins(int* bins, int nb, int* warp_sums, int* carry_s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int base = 0; base < nb; base += 1024) {
    const int i = base + threadIdx.x;
    const int v = i < nb ? bins[i] : 0;
    int incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      int o = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += o;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      int w = warp_sums[lane], wi = w;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        int o = __shfl_up_sync(0xffffffffu, wi, off);
        if (lane >= off) wi += o;
      }
      warp_sums[lane] = wi - w;
    }
    __syncthreads();
    const int excl = *carry_s + warp_sums[warp] + incl - v;
    if (i < nb) bins[i] = excl;
    __syncthreads();
    if (threadIdx.x == 1023) *carry_s = excl + v;
    __syncthreads();
  }
}
// Key of a token in the combine order from `last` = 1 + its largest padded routed row (0: no row).
__device__ __forceinline__ int order_key(int last) { return last == 0 ? 0 : (last - 1) / BLOCK_M + 1; }

// Combine order of the persistent launch: tokens sorted by the M-block of their LAST row in the expert-ordered
// row space (a counting sort; one block).  The operators walk the experts in order, so this is the order in
// which tokens become complete: combine tasks taken in this order find their dependent events met one after
// the other instead of all at the very end.  Tokens without any row come first.
constexpr int ORDER_MAX_BINS = 12000;   // bins (M-blocks + 1) that fit the block's shared memory
__global__ void __launch_bounds__(1024) layout_order_kernel(int T, LayoutView lv) {
  extern __shared__ int bins[];
  __shared__ int carry_s;
  __shared__ int warp_sums[32];
  if (threadIdx.x == 0) carry_s = 0;
  pdl_trigger();
  pdl_wait();
  const int nb = __ldcg(lv.meta) + 1;
  if (nb > ORDER_MAX_BINS) {   // beyond the shared-memory histogram: token order
    for (int t = threadIdx.x; t < T; t += 1024) lv.combine_order[t] = t;
    return;
  }
  for (int i = threadIdx.x; i < nb; i += 1024) bins[i] = 0;
  __syncthreads();
  // sixteen tokens per thread at a time: their keys are read together and kept for the second pass
  constexpr int U = 16;
  int key[U];
  for (int t0 = threadIdx.x; t0 < T; t0 += U * 1024) {
#pragma unroll
    for (int u = 0; u < U; ++u) key[u] = t0 + u * 1024 < T ? __ldcg(lv.tok_last + t0 + u * 1024) : -1;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (key[u] >= 0) atomicAdd(&bins[key[u] = order_key(key[u])], 1);
  }
  __syncthreads();
  scan_bins(bins, nb, warp_sums, &carry_s);
  const bool kept = T <= U * 1024;
  for (int t0 = threadIdx.x; t0 < T; t0 += U * 1024) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (t0 + u * 1024 < T)
        lv.combine_order[atomicAdd(&bins[kept ? key[u] : order_key(__ldcg(lv.tok_last + t0 + u * 1024))], 1)] = t0 + u * 1024;
  }
}

// The whole layout of fewer than LAYOUT_ONE_SLOTS slots in one block: a thread per slot in the first 31 warps, tables
// in shared memory, nothing read back.  Token generation (V3-shaped layer, 64 tokens) spends 8 us here against 45 us
// in the four kernels and the clearing of the counters.  One chunk of the large form would hold 2048 slots, but its three short kernels overlap, and from a
// thousand slots on they are as fast.
__global__ void __launch_bounds__(1024) layout_one_kernel(const int* __restrict__ ids, int n, int T, int k, int kp, int E,
                                                          int Ep, LayoutView lv, int want_order, DevStatus* status,
                                                          int* __restrict__ zero, int nzero) {
  extern __shared__ int sm[];
  __shared__ int totals[SCAN_ROWS][33];
  __shared__ int carry_s;
  const ExpertScan sc = expert_scan_at(sm, Ep);
  int* s_last = sm + expert_scan_ints(Ep);                       // [LAYOUT_ONE_SLOTS] 1 + padded row of the slot
  int* bins = s_last + LAYOUT_ONE_SLOTS;               // [LAYOUT_ONE_SLOTS + 1]
  uint16_t* whist = reinterpret_cast<uint16_t*>(bins + LAYOUT_ONE_SLOTS + 2 + (expert_scan_ints(Ep) & 1));   // [warps in use][ld]
  const int ld = Ep + (Ep & 1);
  const int warps = (n + 31) >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, i = threadIdx.x;
  for (int q = threadIdx.x; q < warps * ld / 2; q += 1024) reinterpret_cast<uint32_t*>(whist)[q] = 0;
  if (i <= LAYOUT_ONE_SLOTS) bins[i] = 0;
  if (i == 0) carry_s = 0;
  pdl_trigger();
  pdl_wait();
  const int e = i < n ? slot_expert(ids, i, k, kp, E) : -1;
  clear_ints(zero, nzero, threadIdx.x, 1024);
  __syncthreads();
  int r = 0;
  if (warp < warps) {
    const uint32_t peers = __match_any_sync(0xffffffffu, e);
    r = __popc(peers & ((1u << lane) - 1u));
    if (e >= 0 && r == 0) whist[warp * ld + e] = (uint16_t)__popc(peers);
  }
  __syncthreads();
  for (int q = threadIdx.x; q < Ep; q += 1024) {
    int run = 0;
#pragma unroll 8
    for (int w = 0; w < warps; ++w) {
      const int c = whist[w * ld + q];
      whist[w * ld + q] = (uint16_t)run;
      run += c;
    }
    sc.counts[q] = run;
  }
  __syncthreads();
  scan_experts(E, Ep, lv, sc, totals);
  if (i < n) {
    int prow = -1;
    if (e >= 0) {
      const int in_expert = whist[warp * ld + e] + r, row = sc.off[e] + in_expert;
      prow = sc.mb[e] * BLOCK_M + in_expert;
      lv.row_of[i] = row;
      lv.src_of[row] = i;
      if (lv.group_start) lv.group_slot[sc.gr[e] * GROUP_ROWS + in_expert] = i;
    } else {
      lv.row_of[i] = -1;
      note(status, /*MOE_ERR_BAD_EXPERT_ID*/ 1, i);
    }
    lv.prow_of[i] = prow;
    s_last[i] = prow + 1;
  }
  expert_tables(Ep, lv, sc);
  if (!want_order) return;
  __syncthreads();
  int key = 0, at = 0;
  if (i < T) {
    int last = 0;
    for (int j = 0; j < k; ++j) last = max(last, s_last[i * kp + j]);
    key = order_key(last);   // at most the number of M-blocks, which is at most n
    at = atomicAdd(&bins[key], 1);
  }
  __syncthreads();
  scan_bins(bins, sc.mb[Ep] + 1, totals[0], &carry_s);
  if (i < T) lv.combine_order[bins[key] + at] = i;
}

// The whole layout of up to LAYOUT_CLUSTER_SLOTS slots in one cluster of C blocks: block b owns the tokens [b tpc, (b + 1) tpc),
// a warp of it G groups of 32 consecutive slots.  Histograms and bins are exchanged through distributed shared memory, so
// nothing is read back from global memory and the four kernels' starts and ends are paid once: 8192 slots take 8 us
// (11 us with the combine order) instead of 13 (19).  A group costs 3 us -- scattered stores and match instructions of one SM --
// so from 8192 slots on there are sixteen blocks, and at 65536 slots, where a block has four groups, the four kernels over
// all SMs catch up.
// M-blocks and one: at most LAYOUT_CLUSTER_SLOTS / 128 + one per expert
constexpr int LAYOUT_CLUSTER_BINS = LAYOUT_CLUSTER_SLOTS / BLOCK_M + LAYOUT_CLUSTER_EXPERTS + 1;
static_assert(LAYOUT_CLUSTER_BINS <= 1024, "a bin per thread");
__device__ __forceinline__ int ld_cluster(const int* p, uint32_t rank) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(map_to_rank(smem_u32(p), rank)) : "memory");
  return v;
}
__host__ __device__ constexpr size_t layout_cluster_smem(int Ep, int G) {
  return sizeof(int) * (size_t)(expert_scan_ints(Ep) + 2 * Ep + 2 * LAYOUT_CLUSTER_BINS + G * 1024 + 1) +
         sizeof(uint16_t) * 32 * (size_t)(Ep + (Ep & 1));
}
template <int C>
__global__ void __launch_bounds__(1024)
    layout_cluster_kernel(const int* __restrict__ ids, int n, int T, int k, int kp, int E, int Ep, int G, LayoutView lv,
                          int want_order, DevStatus* status, int* __restrict__ zero, int nzero) {
  extern __shared__ int sm[];
  __shared__ int totals[SCAN_ROWS][33];
  __shared__ int carry_s;
  const ExpertScan sc = expert_scan_at(sm, Ep);
  int* hist = sm + expert_scan_ints(Ep);        // [Ep] rows of this block's tokens, read by the other blocks
  int* base = hist + Ep;                        // [Ep] rows of the blocks before this one
  int* bins = base + Ep;                        // [bins] this block's tokens by key, read by the other blocks
  int* place = bins + LAYOUT_CLUSTER_BINS;      // [bins] first place of this block's tokens of the key
  int* s_last = place + LAYOUT_CLUSTER_BINS;    // [G * 1024] 1 + padded row of the slot
  uint16_t* whist = reinterpret_cast<uint16_t*>(s_last + G * 1024 + ((expert_scan_ints(Ep) + G * 1024) & 1));   // [32][ld]
  const int ld = Ep + (Ep & 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int tpc = (T + C - 1) / C;
  const int s0 = min(n, rank * tpc * kp), s1 = min(n, s0 + tpc * kp);   // this block's slots
  for (int q = threadIdx.x; q < 32 * ld / 2; q += 1024) reinterpret_cast<uint32_t*>(whist)[q] = 0;
  for (int q = threadIdx.x; q < LAYOUT_CLUSTER_BINS; q += 1024) bins[q] = 0;
  if (threadIdx.x == 0) carry_s = 0;
  pdl_trigger();
  pdl_wait();
  const int i0 = s0 + warp * (G * 32) + lane;
  int e[LAYOUT_CLUSTER_G], r[LAYOUT_CLUSTER_G];
#pragma unroll
  for (int g = 0; g < LAYOUT_CLUSTER_G; ++g) e[g] = g < G && i0 + 32 * g < s1 ? slot_expert(ids, i0 + 32 * g, k, kp, E) : -1;
  clear_ints(zero, nzero, rank * 1024 + threadIdx.x, C * 1024);
  __syncthreads();
  uint16_t* mine = whist + warp * ld;
#pragma unroll
  for (int g = 0; g < LAYOUT_CLUSTER_G; ++g) {
    if (g >= G) break;
    const uint32_t peers = __match_any_sync(0xffffffffu, e[g]);
    r[g] = e[g] >= 0 ? mine[e[g]] + __popc(peers & ((1u << lane) - 1u)) : 0;
    __syncwarp();
    if (e[g] >= 0 && lane == __ffs(peers) - 1) mine[e[g]] += (uint16_t)__popc(peers);
    __syncwarp();
  }
  __syncthreads();
  for (int q = threadIdx.x; q < Ep; q += 1024) {   // per expert: the block's rows in front of each warp's
    int run = 0;
#pragma unroll 8
    for (int w = 0; w < 32; ++w) {
      const int c = whist[w * ld + q];
      whist[w * ld + q] = (uint16_t)run;
      run += c;
    }
    hist[q] = run;
  }
  cluster_sync_all();
  for (int q = threadIdx.x; q < Ep; q += 1024) {
    int c[C], sum = 0;
#pragma unroll
    for (int b = 0; b < C; ++b) c[b] = ld_cluster(hist + q, b);
#pragma unroll
    for (int b = 0; b < C; ++b) {
      if (b == rank) base[q] = sum;
      sum += c[b];
    }
    sc.counts[q] = sum;
  }
  __syncthreads();
  scan_experts(E, Ep, lv, sc, totals, rank == 0);
#pragma unroll
  for (int g = 0; g < LAYOUT_CLUSTER_G; ++g) {
    const int i = i0 + 32 * g;
    if (g >= G || i >= s1) break;
    int prow = -1;
    if (e[g] >= 0) {
      const int in_expert = base[e[g]] + mine[e[g]] + r[g], row = sc.off[e[g]] + in_expert;
      prow = sc.mb[e[g]] * BLOCK_M + in_expert;
      lv.row_of[i] = row;
      lv.src_of[row] = i;
      if (lv.group_start) lv.group_slot[sc.gr[e[g]] * GROUP_ROWS + in_expert] = i;
    } else {
      lv.row_of[i] = -1;
      note(status, /*MOE_ERR_BAD_EXPERT_ID*/ 1, i);   // the slot is dropped, the layer carries on
    }
    lv.prow_of[i] = prow;
    s_last[i - s0] = prow + 1;
  }
  expert_tables(Ep, lv, sc, rank, C);
  if (!want_order) {
    cluster_sync_all();   // no block leaves while another reads its histogram
    return;
  }
  __syncthreads();
  // combine order (layout_order_kernel): a counting sort of the tokens by the M-block of their last routed row
  const int nt = (s1 - s0) / kp;
  int key[LAYOUT_CLUSTER_G], at[LAYOUT_CLUSTER_G];
#pragma unroll
  for (int g = 0; g < LAYOUT_CLUSTER_G; ++g) {
    const int t = threadIdx.x + 1024 * g;
    if (t >= nt) break;
    int last = 0;
    for (int j = 0; j < k; ++j) last = max(last, s_last[t * kp + j]);
    key[g] = order_key(last);
    at[g] = atomicAdd(&bins[key[g]], 1);
  }
  cluster_sync_all();
  const int nb = sc.mb[Ep] + 1;
  int before = 0;
  if ((int)threadIdx.x < nb) {
    int c[C], sum = 0;
#pragma unroll
    for (int b = 0; b < C; ++b) c[b] = ld_cluster(bins + threadIdx.x, b);
#pragma unroll
    for (int b = 0; b < C; ++b) {
      if (b == rank) before = sum;
      sum += c[b];
    }
    place[threadIdx.x] = sum;
  }
  __syncthreads();
  scan_bins(place, nb, totals[0], &carry_s);
  if ((int)threadIdx.x < nb) place[threadIdx.x] += before;
  __syncthreads();
#pragma unroll
  for (int g = 0; g < LAYOUT_CLUSTER_G; ++g) {
    const int t = threadIdx.x + 1024 * g;
    if (t >= nt) break;
    lv.combine_order[place[key[g]] + at[g]] = rank * tpc + t;
  }
  cluster_sync_all();   // no block leaves while another reads its bins
}

// Can the current device hold a cluster of C such blocks?  Looked up once per device, with the kernel's largest shared memory.
template <int C>
static cudaError_t layout_cluster_fits(bool* fits) {
  static std::mutex mu;
  static int known[MAX_DEVICES] = {};   // 1: no, 2: yes
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!known[dev]) {
    const size_t smem = layout_cluster_smem(LAYOUT_CLUSTER_EXPERTS, LAYOUT_CLUSTER_G);
    if ((e = cudaFuncSetAttribute(layout_cluster_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    if (C > 8 && (e = cudaFuncSetAttribute(layout_cluster_kernel<C>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1))) return e;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(1024);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, layout_cluster_kernel<C>, &cfg) != cudaSuccess) {
      cudaGetLastError();   // not a size this device knows
      n = 0;
    }
    known[dev] = n > 0 ? 2 : 1;
  }
  *fits = known[dev] == 2;
  return cudaSuccess;
}

template <int C>
static cudaError_t launch_layout_cluster(const int* ids, const Dims& dm, const LayoutView& lv, bool want_order, int* zero, int nzero,
                                         DevStatus* status, cudaStream_t s) {
  const int Ep = dm.Ep(), cta_slots = (dm.T + C - 1) / C * dm.kp(), G = (cta_slots + 1023) / 1024;
  return launch_dependent_cluster(layout_cluster_kernel<C>, C, dim3(C), dim3(1024), layout_cluster_smem(Ep, G), s, ids, dm.slots(), dm.T,
                                  dm.k, dm.kp(), dm.E, Ep, G, lv, want_order ? 1 : 0, status, zero, nzero);
}

cudaError_t launch_layout(const int* topk_ids, const Dims& dm, const LayoutView& lv, bool want_order, int cap_mblocks,
                          int* zero, int nzero, DevStatus* status, cudaStream_t s, int* launches) {
  const int n = dm.slots(), Ep = dm.Ep(), kp = dm.kp();
  cudaError_t e;
  const int wanted = layout_blocks(dm.T, kp, Ep, true, true);
  if (wanted == 1) {
    const size_t smem = sizeof(int) * (size_t)(expert_scan_ints(Ep) + 4 + 2 * LAYOUT_ONE_SLOTS) +
                        sizeof(uint16_t) * (size_t)((n + 31) / 32) * (Ep + (Ep & 1));
    ++*launches;
    return launch_dependent(layout_one_kernel, dim3(1), dim3(1024), smem, s, topk_ids, n, dm.T, dm.k, kp, dm.E, Ep, lv,
                            want_order ? 1 : 0, status, zero, nzero);
  }
  if (wanted) {
    bool fits = false;
    if ((e = wanted == 8 ? layout_cluster_fits<8>(&fits) : layout_cluster_fits<16>(&fits))) return e;
    const int blocks = layout_blocks(dm.T, kp, Ep, fits, fits);
    if (blocks) ++*launches;
    if (blocks == 8) return launch_layout_cluster<8>(topk_ids, dm, lv, want_order, zero, nzero, status, s);
    if (blocks == 16) return launch_layout_cluster<16>(topk_ids, dm, lv, want_order, zero, nzero, status, s);
  }
  const int nblk = n > 0 ? (n + LAYOUT_CHUNK - 1) / LAYOUT_CHUNK : 1;
  int* const tok_last = want_order ? lv.tok_last : nullptr;
  LayoutView lr = lv;
  lr.tok_last = tok_last;
  if ((e = launch_dependent(layout_hist_kernel, dim3(nblk), dim3(HIST_THREADS), sizeof(int) * (size_t)Ep, s, topk_ids, n, dm.k,
                            kp, dm.E, Ep, lv.blk_hist, tok_last, zero, nzero)))
    return e;
  const int ranges = Ep <= 1024 ? 1024 / Ep : 1;
  if ((e = launch_dependent(layout_scan_kernel, dim3(1), dim3(1024), sizeof(int) * (expert_scan_ints(Ep) + (size_t)ranges * Ep), s, nblk, dm.E, Ep, lv)))
    return e;
  const size_t nlast = LAYOUT_CHUNK / kp + 2;
  auto rank_smem = [&](int warps) {
    return sizeof(int) * (3 * (size_t)Ep + nlast + 1) + sizeof(uint16_t) * (size_t)warps * (Ep + (Ep & 1));
  };
  // as many warps as have room for their histograms in 48 KB of shared memory (32 up to about 500 experts)
  constexpr size_t ROOM = 48 * 1024;
  if (rank_smem(32) <= ROOM)
    e = launch_dependent(layout_rank_kernel<32>, dim3(nblk), dim3(1024), rank_smem(32), s, topk_ids, n, dm.k, kp, dm.E, Ep, lr, status);
  else if (rank_smem(16) <= ROOM)
    e = launch_dependent(layout_rank_kernel<16>, dim3(nblk), dim3(512), rank_smem(16), s, topk_ids, n, dm.k, kp, dm.E, Ep, lr, status);
  else
    e = launch_dependent(layout_rank_kernel<8>, dim3(nblk), dim3(256), rank_smem(8), s, topk_ids, n, dm.k, kp, dm.E, Ep, lr, status);
  if (e) return e;
  *launches += 3;
  if (want_order) {
    int nb = cap_mblocks + 2;
    if (nb > ORDER_MAX_BINS) nb = ORDER_MAX_BINS;
    if ((e = launch_dependent(layout_order_kernel, dim3(1), dim3(1024), sizeof(int) * (size_t)nb, s, dm.T, lv))) return e;
    ++*launches;
  }
  return cudaSuccess;
}

}  // namespace moe

// ------------------------------------------------------------------------------------------
// Dispatch layout without any allocation.
//
// Some callers may not allocate device memory at the point where they need the layout: code
// running inside a framework's memory-planned region or a real-time serving loop where cudaMalloc
// (which synchronises the device and may fail under fragmentation) is forbidden, plugins that are
// handed only their input and output buffers, and callers that never created a moe_ctx.  For them
// the scratch of the layout kernels (per-block histograms, M-block table, padded-row indices,
// status word) lives in the fixed-size array below, which every GPU that loads this library holds
// until the process exits (about 1.6 MB).  All calls share it.
// ------------------------------------------------------------------------------------------
#include <mutex>

#include "../../include/moe_b200.h"

namespace {

constexpr int NA_MAX_SLOTS = MOE_NOALLOC_MAX_SLOTS;             // T * (k + S)
constexpr int NA_MAX_EP = MOE_NOALLOC_MAX_EXPERTS;              // E + S
constexpr int NA_MAX_BLOCKS = NA_MAX_SLOTS / moe::LAYOUT_CHUNK; // blocks of the layout kernels
constexpr int NA_MAX_HIST = 1 << 17;                            // ints of per-block histograms (nblk * (E+S))
constexpr int NA_MAX_MBLK = (NA_MAX_SLOTS + NA_MAX_EP * (moe::BLOCK_M - 1)) / moe::BLOCK_M + 2;

struct NoAllocScratch {
  moe::DevStatus status;
  int meta[8];
  int pad_off[NA_MAX_EP + 1];
  int mb_start[NA_MAX_EP + 1];
  int mblk_expert[NA_MAX_MBLK];
  int work_start[NA_MAX_EP + 1];
  int wblk_expert[NA_MAX_MBLK];
  int blk_hist[NA_MAX_HIST];
  int prow_of[NA_MAX_SLOTS];
};

// In host code this name is only a handle for cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoAllocScratch)];

constexpr int NA_MAX_DEVICES = 64;
std::mutex g_na_mutex;
NoAllocScratch* g_na_ptr[NA_MAX_DEVICES] = {};

}  // namespace

extern "C" int moe_layout_noalloc(const int32_t* topk_ids, int32_t T, int32_t E, int32_t k, int32_t n_shared,
                                  int32_t* counts, int32_t* offsets, int32_t* row_of, int32_t* src_of,
                                  int32_t* status2, void* stream) {
  if (!topk_ids || !counts || !offsets || !row_of || !src_of) return MOE_ERR_INVALID_ARG;
  if (T < 1 || E < 1 || E > 1024 || k < 1 || k > E || n_shared < 0) return MOE_ERR_INVALID_ARG;
  const long slots = (long)T * (k + n_shared);
  const int Ep = E + n_shared;
  const long nblk = (slots + moe::LAYOUT_CHUNK - 1) / moe::LAYOUT_CHUNK;
  if (slots > NA_MAX_SLOTS || Ep > NA_MAX_EP || nblk > NA_MAX_BLOCKS || nblk * Ep > NA_MAX_HIST)
    return MOE_ERR_TOO_LARGE;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) return MOE_ERR_NO_DEVICE;
  NoAllocScratch* sc = nullptr;
  {
    // first call on this device: resolve the device address of the static array (device `dev` is current)
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_ptr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
        cudaGetLastError();
        return MOE_ERR_CUDA;
      }
      g_na_ptr[dev] = static_cast<NoAllocScratch*>(p);
    }
    sc = g_na_ptr[dev];
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  moe::Dims dm{T, 8, E, k, n_shared, 8};
  moe::LayoutView lv{};   // (fields not set below stay NULL: no combine order here)
  lv.counts = counts;
  lv.offsets = offsets;
  lv.row_of = row_of;
  lv.src_of = src_of;
  lv.prow_of = sc->prow_of;
  lv.pad_off = sc->pad_off;
  lv.mb_start = sc->mb_start;
  lv.mblk_expert = sc->mblk_expert;
  lv.work_start = sc->work_start;
  lv.wblk_expert = sc->wblk_expert;
  lv.meta = sc->meta;
  lv.blk_hist = sc->blk_hist;
  int launches = 0;
  // the array keeps the previous call's contents: the first kernel clears the status word
  if (moe::launch_layout(topk_ids, dm, lv, false, 0, reinterpret_cast<int*>(&sc->status), sizeof(moe::DevStatus) / sizeof(int),
                         &sc->status, st, &launches) != cudaSuccess)
    return MOE_ERR_CUDA;
  if (status2 &&
      cudaMemcpyAsync(status2, &sc->status, 2 * sizeof(int), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return MOE_ERR_CUDA;
  return MOE_OK;
}
