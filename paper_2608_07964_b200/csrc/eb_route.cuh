// Gating of one token by one warp.  Lane i holds logits i, i+32, ...  (E <= 256 -> at most 8 per lane).  K rounds of
// a warp arg-max under the order (value descending, index ascending) pick the experts.  The logits are compared as
// integers that order like the floats (-0 counts as 0, as in a float comparison), so the decision is exact and a
// round is two warp reductions (redux) instead of ten shuffles.
#pragma once

#include "eb_dispatch.cuh"

namespace {

constexpr int kMaxPerLane = EB_MAX_E / 32;

// Unsigned integers in the order of the floats; never 0, which stands for "no candidate".
__device__ __forceinline__ unsigned float_key(float v) {
  const unsigned b = __float_as_uint(v + 0.f);   // -0 + 0 = +0
  const unsigned k = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
  return k ? k : 1u;
}
__device__ __forceinline__ float key_float(unsigned k) { return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k); }

// Routes token t (E <= 32 PL): writes its row of topk_idx and topk_w.  Returns expert number `lane` of the token in lanes below K.
template <int PL>
__device__ __forceinline__ int route_token(const ModelParams& mp, int t, int lane, const float* __restrict__ logits,
                                           int32_t* __restrict__ topk_idx, float* __restrict__ topk_w) {
  const int E = mp.E, K = mp.K;
  const float* z = logits + (size_t)t * E;
  float v[PL];
  unsigned key[PL];   // 0: beyond E, or taken
#pragma unroll
  for (int i = 0; i < PL; ++i) v[i] = lane + 32 * i < E ? z[lane + 32 * i] : 0.f;
#pragma unroll
  for (int i = 0; i < PL; ++i) key[i] = lane + 32 * i < E ? float_key(v[i]) : 0u;

  float z_top = 0.f, my_p = 0.f, p_sum = 0.f;
  int my_e = -1;
  for (int k = 0; k < K; ++k) {
    unsigned bk = key[0];
    int bi = 0;
#pragma unroll
    for (int i = 1; i < PL; ++i)
      if (key[i] > bk) {   // ascending i keeps the lower index on ties
        bk = key[i];
        bi = i;
      }
    const unsigned top = __reduce_max_sync(0xffffffffu, bk);
    const int be = (int)__reduce_min_sync(0xffffffffu, bk == top ? (unsigned)(lane + 32 * bi) : 0xffffffffu);
#pragma unroll
    for (int i = 0; i < PL; ++i)
      if (lane + 32 * i == be) key[i] = 0u;
    const float bv = key_float(top);
    if (k == 0) z_top = bv;
    const float p = expf(bv - z_top);
    p_sum += p;
    if (lane == k) {
      my_e = be;
      my_p = p;
    }
  }
  if (!mp.renorm) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < PL; ++i)
      if (lane + 32 * i < E) s += expf(v[i] - z_top);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    p_sum = s;
  }
  if (lane < K) {
    topk_idx[(size_t)t * K + lane] = my_e;
    topk_w[(size_t)t * K + lane] = my_p / p_sum;
  }
  return my_e;
}

constexpr int kChunkThreads = 1024;   // a warp per token of a chunk.  With PL = 2 (E <= 64) the registers leave room for two blocks per SM

// Chunk c of micro-batch j by one block: its tokens are routed (or keep their routing), s_hist [E] gets their assignments per
// expert.  Ends with a block barrier.
template <int PL>
__device__ __forceinline__ void route_chunk(const ModelParams& mp, const BatchParams& bp, int c, int j, bool routed, const float* __restrict__ logits,
                                            int32_t* __restrict__ topk_idx, float* __restrict__ topk_w, int* s_hist) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int e = threadIdx.x; e < mp.E; e += kChunkThreads) s_hist[e] = 0;
  __syncthreads();
  const int t = bp.tok_off[j] + (c - bp.chunk_off[j]) * 32 + warp;
  if (t < bp.tok_off[j + 1]) {
    int e = -1;
    if (routed) e = route_token<PL>(mp, t, lane, logits, topk_idx, topk_w);
    else if (lane < mp.K) e = topk_idx[(size_t)t * mp.K + lane];   // deferred: routed when it reached its layer
    // an index outside [0, E) (only in a table not written by the routing) is skipped here and reported by the dispatch
    if (lane < mp.K && (unsigned)e < (unsigned)mp.E) atomicAdd(&s_hist[e], 1);
  }
  __syncthreads();
}

}  // namespace
