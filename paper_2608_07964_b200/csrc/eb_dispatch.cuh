// Shape of a step as the dispatch kernels see it: active layers, home devices, numbering of the groups.
#pragma once

#include "eb_internal.cuh"

namespace {

struct StepShape {
  int nl;                       // active layers
  int act_layer[EB_MAX_MB];     // ascending
  int rank_of_mb[EB_MAX_MB];    // rank of the micro-batch's layer among active layers, -1 if not chosen
};

// first token (local index) of micro-batch of T tokens whose home device is >= d
__device__ __forceinline__ int home_start(int d, int T, int D) {
  if (T < (1 << 26)) return (int)(((unsigned)d * (unsigned)T + (unsigned)(D - 1)) / (unsigned)D);   // d <= 16: no overflow
  return (int)(((long long)d * T + D - 1) / D);
}
// home device of local token tl of a micro-batch of T tokens: floor(tl * D / T)
__device__ __forceinline__ int home_device(int tl, int T, int D) {
  if (T < (1 << 26)) return (int)(((unsigned)tl * (unsigned)D) / (unsigned)T);
  return (int)(((long long)tl * D) / T);
}

// Active layers of a step and every micro-batch's rank among them: threads 0..15 each place one
// micro-batch, the result lands in shared memory.  Ends with a block barrier.
__device__ __forceinline__ void step_shape_block(const BatchParams& bp, uint32_t run, StepShape* out) {
  const int j = threadIdx.x;
  if (j < 32) {   // warp 0; lanes 0..15 each own one micro-batch
    const bool sel = j < bp.n_mb && ((run >> j) & 1u);
    const int my_layer = j < bp.n_mb ? bp.layer[j] : -1;
    // is j the first chosen micro-batch sitting at its layer?
    const unsigned peers = __match_any_sync(0xffffffffu, sel ? my_layer : -1 - j);
    const bool first = sel && j == __ffs(peers) - 1;
    // distinct chosen layers below mine, and in total
    const unsigned firsts = __ballot_sync(0xffffffffu, first);
    const int total = __popc(firsts);
    int below = 0;
#pragma unroll
    for (int i = 0; i < EB_MAX_MB; ++i) {
      const int li = __shfl_sync(0xffffffffu, my_layer, i);
      below += ((firsts >> i) & 1u) && li < my_layer;
    }
    if (j < EB_MAX_MB) {
      out->rank_of_mb[j] = sel ? below : -1;
      if (first) out->act_layer[below] = my_layer;
      if (j == 0) out->nl = total;
    }
  }
  __syncthreads();
}

// group id of (device d, active-layer rank lr, local slot) ; local slot < n_d + S
__device__ __forceinline__ int group_id(const int* dev_off, int S, int nl, int d, int lr, int local) {
  int n_d = dev_off[d + 1] - dev_off[d];
  return nl * (dev_off[d] + d * S) + lr * (n_d + S) + local;
}

__device__ __forceinline__ int mb_of_chunk(const BatchParams& bp, int c) {
  int j = 0;
  while (j + 1 < bp.n_mb && c >= bp.chunk_off[j + 1]) ++j;
  return j;
}

}  // namespace
