// Router in the path (Section 2.2, first paragraph: the router scores the experts for every token and keeps the
// top k): logits = x W_r^T on the tensor cores with the softmax top-k of route_layout.cu's router fused into the
// epilogue, and the gradient of the k scores with respect to the logits.
//
// Forward: the router weights are the A operand (128 experts per accumulator, two accumulators above 128 experts), a
// tile of up to 256 tokens the B operand, and a cluster of 1, 2, 4 or 8 CTAs shares a tile by splitting the reduction
// over d.  Each CTA streams its k-blocks through a TMA ring into TMEM; then the CTAs exchange partial sums through
// distributed shared memory -- every CTA ends up with all experts' partials for its share of the tile's tokens, adds them in
// CTA order, so the result does not depend on timing -- and its sixteen warps select, four tokens per warp
// (warp_topk: raw logits compared, ties to the lower id, slots in descending order).
//
// What bounds it: few tokens, latency -- W_r is 3.7 MB at 256 x 7168 and one CTA pair needed 65 us to stream it; many tokens,
// the reads of x, if all SMs have a share of them.  Tiles of 256 tokens without a split occupied 64 of 148 SMs on 8192
// tokens, with the selection exposed behind them: 70 us.  See plan_router_fwd for the choice of tile and split.
#include <limits.h>

#include "gemm_tile.cuh"
#include "launch_pairs.cuh"
#include "moe_internal.h"
#include "topk.cuh"

namespace moe {

constexpr int ROUTER_WARPS = 16;      // warp 0 TMA producer, warp 1 MMA issuer and TMEM owner; all of them the epilogue
constexpr int ROUTER_THREADS = 32 * ROUTER_WARPS;
constexpr int ROUTER_MAX_STAGES = 8;
constexpr int ROUTER_W_BYTES = 128 * BK * 2;   // 128 experts of one k-block
constexpr int ROUTER_SMEM_MAX = 222 * 1024;    // operand ring, later the exchanged partial sums
constexpr int ROUTER_MAX_CLUSTER = 8;

struct RouterBarriers {
  uint64_t full[ROUTER_MAX_STAGES], empty[ROUTER_MAX_STAGES];
  uint64_t acc_full;
  uint32_t tmem_base;
};

// Four tokens of one warp: `row` = their logits' partial sums [nslots][..][EPAD experts][4 tokens], added here.
template <int NACC>
__device__ __forceinline__ void router_select(const RouterArgs& a, float4* row, int nslots, size_t slot_stride, int token0,
                                              int lane) {
  constexpr int NPL = 4 * NACC;
  float v[4][NPL];
  uint64_t* pool = reinterpret_cast<uint64_t*>(row);   // the first source's sums, once they are read: 2 or 4 KB
  {
    float4 acc[NPL];
#pragma unroll
    for (int i = 0; i < NPL; ++i) acc[i] = row[i * 32 + lane];
#pragma unroll 1
    for (int r = 1; r < nslots; ++r) {
      row += slot_stride;
      float4 w[NPL];
#pragma unroll
      for (int i = 0; i < NPL; ++i) w[i] = row[i * 32 + lane];
#pragma unroll
      for (int i = 0; i < NPL; ++i) { acc[i].x += w[i].x; acc[i].y += w[i].y; acc[i].z += w[i].z; acc[i].w += w[i].w; }
    }
#pragma unroll
    for (int i = 0; i < NPL; ++i) { v[0][i] = acc[i].x; v[1][i] = acc[i].y; v[2][i] = acc[i].z; v[3][i] = acc[i].w; }
  }
  if (a.logits)
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
      for (int i = 0; i < NPL; ++i)
        if (token0 + t < a.T && i * 32 + lane < a.E) a.logits[(size_t)(token0 + t) * a.E + i * 32 + lane] = v[t][i];
  uint32_t key[4][NPL];
  float mx[4], den[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
#pragma unroll
    for (int i = 0; i < NPL; ++i) key[t][i] = i * 32 + lane < a.E ? float_key(v[t][i]) : 0u;
    mx[t] = key_float(__reduce_max_sync(0xffffffffu, lane_max<NPL>(key[t])));
    den[t] = 0.f;
  }
  if (!(a.renorm & GATE_SIGMOID)) {
#pragma unroll
    for (int i = 0; i < NPL; ++i)
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (i * 32 + lane < a.E) den[t] += expf(v[t][i] - mx[t]);
#pragma unroll
    for (int off = 16; off; off >>= 1)
#pragma unroll
      for (int t = 0; t < 4; ++t) den[t] += __shfl_xor_sync(0xffffffffu, den[t], off);
  }
  int id[4] = {0, 0, 0, 0};
  float l[4] = {0.f, 0.f, 0.f, 0.f}, p[4], wsum[4] = {0.f, 0.f, 0.f, 0.f};
  warp_topk<NPL, 4>(key, a.k, lane, pool, id, l);
#pragma unroll
  for (int t = 0; t < 4; ++t) p[t] = (a.renorm & GATE_SIGMOID) ? 1.0f / (1.0f + expf(-l[t])) : expf(l[t] - mx[t]) / den[t];
  if (a.renorm & GATE_RENORM) {
    for (int j = 0; j < a.k; ++j)
#pragma unroll
      for (int t = 0; t < 4; ++t) wsum[t] += __shfl_sync(0xffffffffu, p[t], j);
#pragma unroll
    for (int t = 0; t < 4; ++t) p[t] /= wsum[t];
  }
  if (lane < a.k)
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (token0 + t < a.T) {
        a.topk_ids[(size_t)(token0 + t) * a.k + lane] = id[t];
        a.topk_w[(size_t)(token0 + t) * a.k + lane] = p[t];
        if (a.counts) atomicAdd(&a.counts[id[t]], 1);
      }
}

template <int NACC>
__global__ void __launch_bounds__(ROUTER_THREADS, 1) router_fwd_kernel(const __grid_constant__ RouterArgs a) {
  constexpr int EPAD = NACC * 128;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ RouterBarriers bars;
  // partial sums of this CTA's tokens, four tokens side by side: [sources but itself (at least one)][token / 4][EPAD][4];
  // behind the operand ring where both fit, in its place (after the k-loop) where they do not
  float4* part = reinterpret_cast<float4*>(smem + (a.part_over_ring ? 0 : a.stages * (NACC * ROUTER_W_BYTES + a.ntok * BK * 2)));

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int C = a.csize, rank = (int)cluster_ctarank();
  const int cluster = blockIdx.x / C, nclusters = gridDim.x / C;
  const WaitCtl wc{a.status, a.budget_ns};
  const int ntok = a.ntok, npc = ntok / C;        // tokens of a tile; tokens this CTA finishes
  const int ntiles = (a.T + ntok - 1) / ntok;
  const int nkb_all = (a.d + BK - 1) / BK;
  const int kb0 = (int)((long)nkb_all * rank / C), kb1 = (int)((long)nkb_all * (rank + 1) / C);
  const int stage_bytes = NACC * ROUTER_W_BYTES + ntok * BK * 2;
  int acc_cols = 32;
  while (acc_cols < ntok) acc_cols <<= 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < a.stages; ++s) {
      mbar_init(&bars.full[s], 1);
      mbar_init(&bars.empty[s], 1);
    }
    mbar_init(&bars.acc_full, 1);
    mbar_fence_init();
    fence_proxy_async();
    tma_prefetch_desc(&a.tmX);
    tma_prefetch_desc(&a.tmW);
  }
  if (warp == 1) {
    tmem_alloc_cta(&bars.tmem_base, NACC * acc_cols);
    tmem_relinquish_cta();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  if (C > 1) cluster_arrive();   // waited for before the first access to another CTA's shared memory
  const uint32_t tmem_base = uniform(bars.tmem_base);
  pdl_trigger();
  pdl_wait();

  uint32_t s_ld = 0, ph_ld = 1, s_mma = 0, ph_mma = 0, n_tile = 0;
  bool ok = true;   // a failed wait: this warp skips the work but still meets the barriers
  for (int t = cluster; t < ntiles; t += nclusters, ++n_tile) {
    const int t0 = t * ntok;
    if (warp == 0) {
      for (int kb = kb0; kb < kb1 && ok; ++kb) {
        if (!mbar_wait_warp(&bars.empty[s_ld], ph_ld, wc, SITE_EMPTY, t, 20)) { ok = false; break; }
        uint8_t* st = smem + s_ld * stage_bytes;
        mbar_expect_tx_elect(&bars.full[s_ld], stage_bytes);
        tma_load_2d(st, &a.tmW, kb * BK, 0, &bars.full[s_ld]);
        if (NACC == 2) tma_load_2d(st + ROUTER_W_BYTES, &a.tmW, kb * BK, 128, &bars.full[s_ld]);
        tma_load_2d(st + NACC * ROUTER_W_BYTES, &a.tmX, kb * BK, t0, &bars.full[s_ld]);
        if (++s_ld == (uint32_t)a.stages) { s_ld = 0; ph_ld ^= 1; }
      }
    } else if (warp == 1) {
      const uint32_t idesc = make_idesc_bf16(BLOCK_M, ntok, 0, 0);
      const uint32_t ring_lo = smem_desc_lo(smem_u32(smem), 16);
      for (int kb = kb0; kb < kb1 && ok; ++kb) {
        if (!mbar_wait_warp(&bars.full[s_mma], ph_mma, wc, SITE_FULL, t)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t w_lo = ring_lo + s_mma * (stage_bytes >> 4), x_lo = w_lo + NACC * (ROUTER_W_BYTES >> 4);
#pragma unroll
        for (int h = 0; h < NACC; ++h)
          tc_mma4_bf16_cta(tmem_base + h * acc_cols, w_lo + h * (ROUTER_W_BYTES >> 4), x_lo, smem_desc_hi(1024), idesc, kb != kb0);
        tc_commit_cta(&bars.empty[s_mma]);
        if (++s_mma == (uint32_t)a.stages) { s_mma = 0; ph_mma ^= 1; }
      }
      tc_commit_cta(&bars.acc_full);   // also after a failed wait: what was issued has completed once this arrives
    }
    __syncwarp();
    int up = 1;
    if (lane == 0) up = mbar_wait(&bars.acc_full, n_tile & 1, wc, SITE_TMEM_FULL, t, 100) ? 1 : 0;
    if (!__shfl_sync(0xffffffffu, up, 0)) ok = false;
    tc_fence_after_sync();
    if (C > 1) {
      if (n_tile == 0) cluster_wait();            // every CTA of the cluster runs
      if (a.part_over_ring) cluster_sync_all();   // every CTA's MMAs are complete: the operand rings may be overwritten
    } else if (a.part_over_ring) {
      __syncthreads();
    }
    // ---- warp w reads TMEM lanes 32 (w % 4) ..: 32 experts; chunks of 16 tokens are dealt to the four warps of a quad.
    // A lane writes four tokens of its expert at a time: 512 contiguous bytes per warp and store.
    const int quad = warp & 3, sub = warp >> 2;
    const uint32_t trow = tmem_base + ((uint32_t)(quad * 32) << 16);
    const int nchunks = ntok / 16, ngroups = npc / 4;
    const size_t slot_stride = (size_t)ngroups * EPAD;
    const int own0 = rank * npc, own1 = own0 + npc;
    const uint32_t part_addr = smem_u32(part);
    // each CTA begins with the next CTA's tokens: in one order they all wrote to the same CTA at a time, and 8192 tokens x
    // 256 experts, d = 7168, with the score gradient took 56.9 us instead of 54.0
    const int first = (rank + 1 < C ? own1 : 0) / 16;
    for (int q = sub; q < nchunks * NACC && C > 1; q += 4) {
      const int h = q / nchunks, cq = q - h * nchunks + first;
      const int c0 = (cq < nchunks ? cq : cq - nchunks) * 16, e = h * 128 + quad * 32 + lane;
      if (c0 >= own0 && c0 + 16 <= own1) continue;   // all of them this CTA's own
      float v[16];
      tmem_ld16(trow + h * acc_cols + c0, v);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 16; i += 4) {
        const int dst = (c0 + i) / npc;
        if (dst == rank) continue;
        const size_t slot = rank < dst ? rank : rank - 1;
        const uint32_t at = (uint32_t)((slot * slot_stride + (size_t)((c0 + i - dst * npc) / 4) * EPAD + e) * 16);
        st_cluster_v4(map_to_rank(part_addr + at, dst), make_uint4(__float_as_uint(v[i]), __float_as_uint(v[i + 1]),
                                                                   __float_as_uint(v[i + 2]), __float_as_uint(v[i + 3])));
      }
    }
    if (C > 1) cluster_sync_all();   // the partial sums of all CTAs have arrived
    for (int q = sub; q < nchunks * NACC; q += 4) {   // this CTA's own, added to the first source's
      const int h = q / nchunks, c0 = (q - h * nchunks) * 16, e = h * 128 + quad * 32 + lane;
      if (c0 >= own1 || c0 + 16 <= own0) continue;
      float v[16];
      tmem_ld16(trow + h * acc_cols + c0, v);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 16; i += 4) {
        const int j = c0 + i - own0;
        if (j < 0 || j >= npc) continue;
        float4* p = part + (size_t)(j / 4) * EPAD + e;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        if (C > 1) s = *p;
        *p = make_float4(s.x + v[i], s.y + v[i + 1], s.z + v[i + 2], s.w + v[i + 3]);
      }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (ok)
      for (int g = warp; g < ngroups; g += ROUTER_WARPS)
        if (t0 + own0 + 4 * g < a.T)
          router_select<NACC>(a, part + (size_t)g * EPAD, C > 1 ? C - 1 : 1, slot_stride, t0 + own0 + 4 * g, lane);
    fence_proxy_async_smem();   // this tile's accesses to the ring's memory before the next tile's loads
    if (t + nclusters < ntiles) cluster_sync_all();
  }

  // ---------------------------------------------------------------- teardown (nobody touches another CTA's memory any more)
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc_cta(tmem_base, NACC * acc_cols);
  }
}

// Co-resident clusters of each size (SMs pair up inside a GPC, so fewer than SMs / size): a property of kernel and device.
struct RouterDevice {
  std::mutex mu;
  bool ready[MAX_DEVICES] = {};
  int clusters[MAX_DEVICES][2][4];   // [accumulators - 1][log2 of the cluster size]
};
static RouterDevice& router_device() { static RouterDevice r; return r; }

static void router_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, int csize, int ctas, size_t smem, cudaStream_t s) {
  memset(cfg, 0, sizeof *cfg);
  cfg->gridDim = dim3(ctas);
  cfg->blockDim = dim3(ROUTER_THREADS);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csize;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 2;
}

// Tile and split.  A CTA's time is the operand bytes it takes in: k-blocks x (expert rows + token rows of a tile), plus, per
// tile, the exchange and selection (charged as ROUTER_TILE_COST rows).  With Q clusters of C CTAs co-resident, the tokens
// are spread evenly over them in as few rounds as 256-token tiles allow.  8192 tokens x 256 experts, d = 7168: C = 4, tiles of
// 240 tokens; 64 tokens: C = 8, tiles of 16.
constexpr int ROUTER_TILE_COST = 1024;
cudaError_t plan_router_fwd(RouterArgs& a, int num_sms) {
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  RouterDevice& rd = router_device();
  {
    std::lock_guard<std::mutex> lock(rd.mu);
    if (!rd.ready[dev]) {
      const int smem = ROUTER_SMEM_MAX + 1024;
      if ((err = cudaFuncSetAttribute(router_fwd_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))) return err;
      if ((err = cudaFuncSetAttribute(router_fwd_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))) return err;
      for (int h = 0; h < 2; ++h)
        for (int q = 0; q < 4; ++q) {
          cudaLaunchConfig_t cfg;
          cudaLaunchAttribute attr[2];
          router_config(&cfg, attr, 1 << q, (num_sms >> q) << q, smem, nullptr);
          cfg.numAttrs = 1;
          int n = 0;
          err = h ? cudaOccupancyMaxActiveClusters(&n, router_fwd_kernel<2>, &cfg) : cudaOccupancyMaxActiveClusters(&n, router_fwd_kernel<1>, &cfg);
          if (err != cudaSuccess) return err;
          rd.clusters[dev][h][q] = n > 0 ? n : 1;
        }
      rd.ready[dev] = true;
    }
  }
  const int nacc = a.E > 128 ? 2 : 1, nkb = (a.d + BK - 1) / BK;
  long best = -1;
  for (int q = 0; q < 4; ++q) {
    const int C = 1 << q, Q = rd.clusters[dev][nacc - 1][q];
    if (C > nkb) break;   // every CTA needs a k-block
    // tile: at most 256 tokens, and the partial sums a CTA receives (its own tokens' if it is alone) fit the ring's memory
    int most = 256;
    while ((long)(C > 1 ? C - 1 : 1) * (most / C) * nacc * 512 > ROUTER_SMEM_MAX) most -= 32;
    const int rounds = (int)(((long)a.T + (long)Q * most - 1) / ((long)Q * most));
    int ntok = (int)(((long)a.T + (long)Q * rounds - 1) / ((long)Q * rounds));
    const int grain = C == 8 ? 32 : 16;   // the MMA's granularity, and four tokens per CTA
    ntok = (ntok + grain - 1) / grain * grain;
    const int tiles = (a.T + ntok - 1) / ntok;
    const long cost = (long)((tiles + Q - 1) / Q) * ((long)((nkb + C - 1) / C) * (nacc * 128 + ntok) + ROUTER_TILE_COST);
    if (best < 0 || cost < best) { best = cost; a.csize = C; a.ntok = ntok; }
  }
  const int stage = nacc * ROUTER_W_BYTES + a.ntok * BK * 2;
  const int per_cta = (nkb + a.csize - 1) / a.csize;
  a.stages = ROUTER_SMEM_MAX / stage;
  if (a.stages > ROUTER_MAX_STAGES) a.stages = ROUTER_MAX_STAGES;
  if (a.stages > per_cta) a.stages = per_cta;
  const int sums = (a.csize > 1 ? a.csize - 1 : 1) * (a.ntok / a.csize) * nacc * 512;
  a.part_over_ring = a.stages * stage + sums > ROUTER_SMEM_MAX;
  a.smem_bytes = 1024 + (a.part_over_ring ? (sums > a.stages * stage ? sums : a.stages * stage) : a.stages * stage + sums);
  return cudaSuccess;
}

cudaError_t launch_router_fwd(const RouterArgs& a, int num_sms, cudaStream_t s, int* launches) {
  if (a.T == 0) return cudaSuccess;
  if (a.counts) {
    cudaError_t e = cudaMemsetAsync(a.counts, 0, sizeof(int) * (size_t)a.E, s);
    if (e != cudaSuccess) return e;
  }
  ++*launches;
  const int tiles = (a.T + a.ntok - 1) / a.ntok;
  int q = 0;
  while ((1 << q) < a.csize) ++q;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const int Q = router_device().clusters[dev][a.E > 128 ? 1 : 0][q];
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  router_config(&cfg, attr, a.csize, (tiles < Q ? tiles : Q) * a.csize, a.smem_bytes, s);
  return a.E > 128 ? cudaLaunchKernelEx(&cfg, router_fwd_kernel<2>, a) : cudaLaunchKernelEx(&cfg, router_fwd_kernel<1>, a);
}

// ------------------------------------------------------------------------------------------
// Backward of the scores: one warp per token, expert e on lane e % 32.  p = softmax(logits) over all E.
//   no renormalisation: dl[e] = [e = e_j] g_j p[e] - p[e] * sum_j g_j p[e_j]
//   renormalisation   : w = softmax over the selected experts; dl[e_j] = w_j (g_j - sum_i g_i w_i), 0 elsewhere
// The selection passes no gradient.
// ------------------------------------------------------------------------------------------
// NPL logits per lane stay in registers (E <= 32 NPL): one read of the logits, one write of the gradient.
template <int NPL>
__global__ void __launch_bounds__(256) router_bwd_kernel(const float* __restrict__ logits, const int* __restrict__ ids,
                                                          const float* __restrict__ g, int T, int E, int k, int mode,
                                                          float* __restrict__ dlogits) {
  const int lane = threadIdx.x & 31;
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  pdl_wait();
  pdl_trigger();
  if (t >= T) return;
  const float* l = logits + (size_t)t * E;
  float* dl = dlogits + (size_t)t * E;
  float v[NPL];
#pragma unroll
  for (int i = 0; i < NPL; ++i) v[i] = i * 32 + lane < E ? l[i * 32 + lane] : -INFINITY;
  // the k selected experts, one per lane (k <= 32)
  const int my_id = lane < k ? ids[(size_t)t * k + lane] : -1;
  const bool have = my_id >= 0 && my_id < E;
  const float my_g = have ? g[(size_t)t * k + lane] : 0.f;
  const float my_l = have ? l[my_id] : 0.f;
  const bool renorm = (mode & GATE_RENORM) != 0;
  if (mode & GATE_SIGMOID) {
    // per-expert scores s = sigmoid(l): only the selected experts get a gradient
    const float s = have ? 1.0f / (1.0f + expf(-my_l)) : 0.f;
    float Z = s;
#pragma unroll
    for (int off = 16; off; off >>= 1) Z += __shfl_xor_sync(0xffffffffu, Z, off);
    float dot = renorm ? my_g * (s / Z) : 0.f;
#pragma unroll
    for (int off = 16; off; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
#pragma unroll
    for (int i = 0; i < NPL; ++i)
      if (i * 32 + lane < E) dl[i * 32 + lane] = 0.f;
    __syncwarp();
    if (have) dl[my_id] = renorm ? s * (1.0f - s) / Z * (my_g - dot) : my_g * s * (1.0f - s);
    return;
  }
  float mx = -INFINITY;
#pragma unroll
  for (int i = 0; i < NPL; ++i) mx = fmaxf(mx, v[i]);
#pragma unroll
  for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  const float my_ex = have ? expf(my_l - mx) : 0.f;
  float den = 0.f;
  if (renorm) {
    den = my_ex;
  } else {
#pragma unroll
    for (int i = 0; i < NPL; ++i)
      if (i * 32 + lane < E) { v[i] = expf(v[i] - mx); den += v[i]; }
  }
#pragma unroll
  for (int off = 16; off; off >>= 1) den += __shfl_xor_sync(0xffffffffu, den, off);
  const float my_w = my_ex / den;
  float dot = my_g * my_w;
#pragma unroll
  for (int off = 16; off; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
  // dense part
#pragma unroll
  for (int i = 0; i < NPL; ++i)
    if (i * 32 + lane < E) dl[i * 32 + lane] = renorm ? 0.f : -(v[i] / den) * dot;
  __syncwarp();
  // the selected experts are distinct, so each lane corrects its own entry
  if (have) dl[my_id] = renorm ? my_w * (my_g - dot) : my_w * my_g - my_w * dot;
}

cudaError_t launch_router_bwd(const float* logits, const int* ids, const float* g, int T, int E, int k, int gate_mode,
                              float* dlogits, cudaStream_t s, int* launches) {
  if (T == 0) return cudaSuccess;
  const dim3 threads(256), grid((T + 7) / 8);
  const int npl = (E + 31) / 32;
  cudaError_t e;
#define MOE_ROUTER_BWD_CASE(N) e = launch_dependent(router_bwd_kernel<N>, grid, threads, 0, s, logits, ids, g, T, E, k, gate_mode, dlogits)
  if (npl <= 1) MOE_ROUTER_BWD_CASE(1);
  else if (npl <= 2) MOE_ROUTER_BWD_CASE(2);
  else if (npl <= 4) MOE_ROUTER_BWD_CASE(4);
  else if (npl <= 8) MOE_ROUTER_BWD_CASE(8);
  else if (npl <= 16) MOE_ROUTER_BWD_CASE(16);
  else MOE_ROUTER_BWD_CASE(32);
#undef MOE_ROUTER_BWD_CASE
  ++*launches;
  return e;
}

}  // namespace moe
