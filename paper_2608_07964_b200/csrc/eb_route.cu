// eb_route: top-k softmax gating (Section 2.1) and per-micro-batch workload vectors (Section 2.3).
//
// One warp per token, a block per chunk of at most 32 tokens of one micro-batch (eb_route.cuh).  Loads are integer counts:
// gathered per block in shared memory, then added with integer atomics in global memory (order independent, hence
// deterministic); a clearing kernel zeroes the rows of the micro-batches being routed first.  What bounds many tokens over few
// experts is those atomics, all on the same few words: added token by token, 16 x 4096 tokens to one of 8 experts took 64 us
// and 1 x 4096 to 6 of 64 19; per chunk 22 and 11.
#include "eb_route.cuh"

namespace {

template <int PL>
__global__ void __launch_bounds__(kChunkThreads, PL <= 2 ? 2 : 1)
route_kernel(ModelParams mp, BatchParams bp, uint32_t route_mask, const float* __restrict__ logits,
             int32_t* __restrict__ topk_idx, float* __restrict__ topk_w, int32_t* __restrict__ mb_load,
             int32_t* __restrict__ mb_cnt) {
  EB_GRID_DEP_SYNC();
  __shared__ int s_hist[EB_MAX_E], s_load[EB_MAX_D];
  const int c = blockIdx.x, j = mb_of_chunk(bp, c), tid = threadIdx.x;
  if (!((route_mask >> j) & 1u)) return;
  if (tid < mp.D) s_load[tid] = 0;
  route_chunk<PL>(mp, bp, c, j, true, logits, topk_idx, topk_w, s_hist);
  if (tid < mp.E && s_hist[tid] > 0) {
    atomicAdd(&mb_cnt[j * mp.E + tid], s_hist[tid]);
    atomicAdd(&s_load[mp.e2d[tid]], s_hist[tid]);
  }
  __syncthreads();
  if (tid < mp.D && s_load[tid] > 0) atomicAdd(&mb_load[j * mp.D + tid], s_load[tid]);
}

__global__ void route_clear_kernel(ModelParams mp, BatchParams bp, uint32_t route_mask, int32_t* mb_load,
                                   int32_t* mb_cnt) {
  EB_GRID_DEP_SYNC();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int per = mp.E + mp.D;
  if (i >= bp.n_mb * per) return;
  int j = i / per, r = i % per;
  if (!((route_mask >> j) & 1u)) return;
  if (r < mp.E) mb_cnt[j * mp.E + r] = 0;
  else mb_load[j * mp.D + (r - mp.E)] = 0;
}

}  // namespace

extern "C" eb_status eb_route(eb_ctx* c, void* stream, const eb_batch* batch, uint32_t route_mask,
                              const float* logits, int32_t* topk_idx, float* topk_w, int32_t* mb_load,
                              int32_t* mb_cnt) {
  if (!c) return EB_ERR_INVALID_ARG;
  BatchParams bp;
  eb_status s = ebi_make_batch(c, batch, &bp);
  if (s != EB_OK) return s;
  if (!logits || !topk_idx || !topk_w || !mb_load || !mb_cnt) return ebi_fail(c, EB_ERR_INVALID_ARG, "null pointer");
  if (bp.n_mb < 32 && (route_mask >> bp.n_mb) != 0) return ebi_fail(c, EB_ERR_INVALID_ARG, "route_mask beyond n_mb");
  if (bp.n_mb == 0 || route_mask == 0) return EB_OK;
  cudaStream_t st = (cudaStream_t)stream;
  KernelTimer timer(c, EBK_ROUTE, st);
  int n = bp.n_mb * (c->cfg.E + c->cfg.D);
  EB_LAUNCH(c, "route", ebi_launch(route_clear_kernel, dim3((n + 255) / 256), dim3(256), 0, st, c->mp, bp, route_mask, mb_load, mb_cnt));
  if (bp.n_chunks > 0)
    EB_LAUNCH(c, "route", ebi_launch(c->cfg.E <= 64 ? route_kernel<2> : route_kernel<kMaxPerLane>, dim3(bp.n_chunks), dim3(kChunkThreads), 0, st,
                                     c->mp, bp, route_mask, logits, topk_idx, topk_w, mb_load, mb_cnt));
  EB_LAUNCH_CHECK(c, "route");
  return EB_OK;
}
