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

// The k largest of the warp's keys: expert e = 32 i + lane in key[i] (0: no expert).  Lane j < k ends up with the j-th
// expert's id and logit; equal logits go to the lower id.  One round is a local argmax and two warp reductions
// (redux), against ten shuffles for a butterfly over {value, id}: the router over 16384 x 128 logits took 34 us with
// the butterfly, its rounds being a serial chain.
template <int NPL>
__device__ __forceinline__ void warp_topk(uint32_t (&key)[NPL], int k, int lane, int* my_id, float* my_logit) {
  for (int j = 0; j < k; ++j) {
    uint32_t bk = key[0];
    int bi = 0;
#pragma unroll
    for (int i = 1; i < NPL; ++i)
      if (key[i] > bk) { bk = key[i]; bi = i; }
    const uint32_t m = __reduce_max_sync(0xffffffffu, bk);
    const int id = __reduce_min_sync(0xffffffffu, bk == m ? bi * 32 + lane : INT_MAX);
    if ((id & 31) == lane) {
#pragma unroll
      for (int i = 0; i < NPL; ++i)
        if (i == (id >> 5)) key[i] = 0;
    }
    if (lane == j) { *my_id = id; *my_logit = key_float(m); }
  }
}

// Programmatic dependent launch.  A kernel launched with launch_dependent() may start while the kernel in front of it
// on the stream still runs; it touches global memory only after pdl_wait(), which returns when that kernel has
// completed.  pdl_trigger() lets the next such kernel start.  Between the layout kernels, each a few microseconds
// long, the launch gap was 2 us.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace moe
