// eb_route: top-k softmax gating (Section 2.1) and per-micro-batch workload vectors (Section 2.3).
//
// One warp per token (eb_route.cuh).
// Loads are integer counts added with integer atomics in global memory (order independent, hence
// deterministic); a clearing kernel zeroes the rows of the micro-batches being routed first.  (Gathering
// the counts per block in shared memory was tried: it needs several tokens per block to pay, and the lost
// parallelism cost more than the atomics it saved.)
#include "eb_route.cuh"

namespace {

constexpr int kWarpsPerBlock = 8;

template <int PL>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
route_kernel(ModelParams mp, BatchParams bp, uint32_t route_mask, const float* __restrict__ logits,
             int32_t* __restrict__ topk_idx, float* __restrict__ topk_w, int32_t* __restrict__ mb_load,
             int32_t* __restrict__ mb_cnt) {
  EB_GRID_DEP_SYNC();
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int t = blockIdx.x * kWarpsPerBlock + warp;
  if (t >= bp.n_tok) return;
  int j = 0;
  while (j + 1 < bp.n_mb && t >= bp.tok_off[j + 1]) ++j;
  if (!((route_mask >> j) & 1u)) return;
  const int my_e = route_token<PL>(mp, t, lane, logits, topk_idx, topk_w);
  if (lane < mp.K) {
    atomicAdd(&mb_cnt[j * mp.E + my_e], 1);
    atomicAdd(&mb_load[j * mp.D + mp.e2d[my_e]], 1);
  }
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
  if (bp.n_tok > 0) {
    int blocks = (bp.n_tok + kWarpsPerBlock - 1) / kWarpsPerBlock;
    EB_LAUNCH(c, "route", ebi_launch(c->cfg.E <= 64 ? route_kernel<2> : route_kernel<kMaxPerLane>, dim3(blocks), dim3(kWarpsPerBlock * 32), 0, st,
                                     c->mp, bp, route_mask, logits, topk_idx, topk_w, mb_load, mb_cnt));
  }
  EB_LAUNCH_CHECK(c, "route");
  return EB_OK;
}
