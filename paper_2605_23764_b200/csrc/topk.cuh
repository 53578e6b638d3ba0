// Warp-wide selection of the k largest logits of a token (shared by the two routers), and the launch helpers of the
// small dependent kernels in front of the layer.
#pragma once

#include <cuda_runtime.h>
#include <limits.h>
#include <stdint.h>
#include <string.h>

namespace moe {

// Order-preserving map of fp32 to uint32: a > b as floats iff key(a) > key(b); the two zeros share a key (raw
// comparison of logits holds them equal), every logit's key is above 0.
__device__ __forceinline__ uint32_t float_key(float x) {
  const uint32_t u = __float_as_uint(x + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t key) {
  return __uint_as_float((key & 0x80000000u) ? (key & 0x7FFFFFFFu) : ~key);
}

template <int NPL>
__device__ __forceinline__ uint32_t lane_max(const uint32_t (&key)[NPL]) {
  uint32_t b[NPL];
#pragma unroll
  for (int i = 0; i < NPL; ++i) b[i] = key[i];
#pragma unroll
  for (int w = 1; w < NPL; w <<= 1)
#pragma unroll
    for (int i = 0; i + w < NPL; i += 2 * w) b[i] = max(b[i], b[i + w]);
  return b[0];
}

// The k largest of each of NT tokens' keys: expert e = 32 i + lane in key[t][i] (0: no expert).  Lane j < k ends up with the
// j-th expert's id and logit of every token; equal logits go to the lower id.
//
// Rounds over all keys: one round is a local argmax -- a tree of depth log2 NPL -- and two warp reductions (redux), against
// ten shuffles for a butterfly over {value, id}; the rounds are a serial chain, so NT tokens side by side hide each other's
// latency.  16384 x 128 logits: 34 us with the butterfly.
template <int NPL, int NT>
__device__ __forceinline__ void warp_topk_rounds(uint32_t (&key)[NT][NPL], int k, int lane, int (&my_id)[NT], float (&my_logit)[NT]) {
#pragma unroll 1
  for (int j = 0; j < k; ++j) {
    uint32_t m[NT];
    int id[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) m[t] = lane_max<NPL>(key[t]);
#pragma unroll
    for (int t = 0; t < NT; ++t) m[t] = __reduce_max_sync(0xffffffffu, m[t]);
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      int c = INT_MAX;
#pragma unroll
      for (int i = NPL - 1; i >= 0; --i) c = key[t][i] == m[t] ? i * 32 + lane : c;   // the lowest id of this lane
      id[t] = c;
    }
#pragma unroll
    for (int t = 0; t < NT; ++t) id[t] = __reduce_min_sync(0xffffffffu, id[t]);
#pragma unroll
    for (int t = 0; t < NT; ++t) {
#pragma unroll
      for (int i = 0; i < NPL; ++i) key[t][i] = id[t] == i * 32 + lane ? 0u : key[t][i];
      my_id[t] = lane == j ? id[t] : my_id[t];
      my_logit[t] = lane == j ? key_float(m[t]) : my_logit[t];
    }
  }
}

// The rounds are bound by the integer pipe, which takes a compare or a select every other cycle (5.6 per key and round).  So
// they go over one key a lane, its largest: the k-th largest of those, taken as the k-th distinct one, is at most the
// k-th largest of all, and about k + 1 to 1.3 k of a token's keys reach it.  These go to shared memory, `pool` (32 entries a
// token, the calling warp's own), in any order, and each finds its rank by comparing {key, ~id} with all of them.  From eight
// keys a lane on (with four, 8 tokens through a V2-Lite layer took 1 % longer); up to k = 16, beyond which more than 32 keys of
// 256 would often reach the bound.  Where they do (many equal logits), or fewer than k do, the rounds take all keys.  Router of
// 8192 tokens x 256 experts, k = 8, with the score gradient: 54.0 -> 52.4 us.
constexpr int TOPK_POOL = 32;
template <int NPL, int NT>
__device__ __forceinline__ void warp_topk(uint32_t (&key)[NT][NPL], int k, int lane, uint64_t* pool, int (&my_id)[NT],
                                          float (&my_logit)[NT]) {
  if constexpr (NPL >= 8) {
    if (k <= 16) {
      uint32_t top[NT], bound[NT];
#pragma unroll
      for (int t = 0; t < NT; ++t) { top[t] = lane_max<NPL>(key[t]); bound[t] = 0; }
#pragma unroll 1
      for (int j = 0; j < k; ++j) {
#pragma unroll
        for (int t = 0; t < NT; ++t) bound[t] = __reduce_max_sync(0xffffffffu, top[t]);
#pragma unroll
        for (int t = 0; t < NT; ++t) top[t] = top[t] == bound[t] ? 0u : top[t];
      }
      __syncwarp();   // the pool's memory has been read as what it was before
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        pool[t * TOPK_POOL + lane] = 0;
        bound[t] = max(bound[t], 1u);
      }
      __syncwarp();
      const uint32_t below = (1u << lane) - 1u;
      int n[NT], least = INT_MAX, most = 0;
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        n[t] = 0;
#pragma unroll
        for (int i = 0; i < NPL; ++i) {
          const bool in = key[t][i] >= bound[t];
          const uint32_t all = __ballot_sync(0xffffffffu, in);
          const int at = n[t] + __popc(all & below);
          if (in && at < TOPK_POOL) pool[t * TOPK_POOL + at] = ((uint64_t)key[t][i] << 32) | (uint32_t)~(i * 32 + lane);
          n[t] += __popc(all);
        }
        least = min(least, n[t]);
        most = max(most, n[t]);
      }
      __syncwarp();
      if (least >= k && most <= TOPK_POOL) {
        uint64_t mine[NT];
        int rank[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t) { mine[t] = pool[t * TOPK_POOL + lane]; rank[t] = 0; }
#pragma unroll 2
        for (int c = 0; c < most; ++c)
#pragma unroll
          for (int t = 0; t < NT; ++t) rank[t] += pool[t * TOPK_POOL + c] > mine[t] ? 1 : 0;
        __syncwarp();
#pragma unroll
        for (int t = 0; t < NT; ++t)
          if (lane < n[t]) pool[t * TOPK_POOL + rank[t]] = mine[t];
        __syncwarp();
#pragma unroll
        for (int t = 0; t < NT; ++t)
          if (lane < k) {
            const uint64_t w = pool[t * TOPK_POOL + lane];
            my_id[t] = (int)~(uint32_t)w;
            my_logit[t] = key_float((uint32_t)(w >> 32));
          }
        return;
      }
    }
  }
  warp_topk_rounds<NPL, NT>(key, k, lane, my_id, my_logit);
}

// Programmatic dependent launch.  A kernel launched with launch_dependent() may start while the kernel in front of it
// on the stream still runs; it touches global memory only after pdl_wait(), which returns when that kernel has
// completed.  pdl_trigger() lets the next such kernel start.  Between the layout kernels, each a few microseconds
// long, the launch gap was 2 us.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_dependent_cluster(void (*kernel)(P...), int csize, dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = csize;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = csize > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <class... P, class... A>
cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  return launch_dependent_cluster(kernel, 1, grid, block, smem, s, args...);
}

}  // namespace moe
