// eb_schedule: Schedule(S, m) of Algorithm 1 (eb_schedule.cuh) as a kernel of its own, one thread block, or several
// for MaxUtil over a large pool.
#include "eb_schedule.cuh"

namespace {

constexpr int kMaxBlocks = 1 << (EB_MAX_MB - 13);

__global__ void __launch_bounds__(kSchedThreads)
schedule_kernel(int D, int n_mb, uint32_t pool_mask, int m, int policy, const int32_t* __restrict__ mb_load,
                eb_sched_result* __restrict__ res, Cand* __restrict__ block_best, unsigned* __restrict__ block_counter) {
  EB_GRID_DEP_SYNC();
  __shared__ SchedShared s;
  __shared__ bool s_last;
  const int tid = threadIdx.x;
  if (tid < EB_MAX_MB * EB_MAX_D) {
    const int j = tid / EB_MAX_D, d = tid % EB_MAX_D;
    s.load[j][d] = (j < n_mb && d < D) ? mb_load[j * D + d] : 0;
  }
  __syncthreads();
  if (!schedule_block(s, D, pool_mask, m, policy, blockIdx.x, gridDim.x)) {
    // every block leaves its best candidate in global memory; the block that arrives last reduces them
    if (tid == 0) {
      block_best[blockIdx.x] = s.best[0];
      __threadfence();
      const unsigned arrived = atomicAdd(block_counter, 1u);
      s_last = arrived == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid < 32) {
      Cand b;
      b.n = -1; b.num = 0; b.peak = 1; b.sub = 0;
      for (int i = tid; i < (int)gridDim.x; i += 32) {
        const Cand o = block_best[i];
        if (better(o, b)) b = o;
      }
      b = warp_best(b);
      const uint32_t mask = run_mask_of(s.member, __popc(pool_mask), b);
      if (tid == 0) {
        s.run = mask;
        *block_counter = 0;   // ready for the next call
      }
    }
    __syncthreads();
  }
  if (tid < 32) write_schedule(s, D, pool_mask, res);
}

}  // namespace

extern "C" eb_status eb_schedule(eb_ctx* c, void* stream, const eb_batch* batch, int32_t m, eb_policy policy,
                                 const int32_t* mb_load, eb_sched_result* d_res, eb_sched_result* h_res) {
  if (!c) return EB_ERR_INVALID_ARG;
  BatchParams bp;
  eb_status s = ebi_make_batch(c, batch, &bp);
  if (s != EB_OK) return s;
  if (!mb_load || !d_res) return ebi_fail(c, EB_ERR_INVALID_ARG, "null pointer");
  if (m < 1) return ebi_fail(c, EB_ERR_INVALID_ARG, "m must be at least 1");
  if ((int)policy < 0 || (int)policy > EB_POLICY_ALL) return ebi_fail(c, EB_ERR_INVALID_ARG, "unknown policy");
  cudaStream_t st = (cudaStream_t)stream;
  {
    // MaxUtil over a large pool: a block per 32 high halves of the subsets; everything else is one block
    int np = 0;
    for (int j = 0; j < bp.n_mb; ++j) np += (batch->pool_mask >> j) & 1u;
    const int blocks = policy == EB_POLICY_MAXUTIL && np > m && np > 13 ? 1 << (np - 13) : 1;
    KernelTimer timer(c, EBK_SCHEDULE, st);
    EB_LAUNCH(c, "schedule", ebi_launch(schedule_kernel, dim3(blocks), dim3(kSchedThreads), 0, st, c->cfg.D, bp.n_mb, batch->pool_mask, (int)m,
                                        (int)policy, mb_load, d_res, (Cand*)c->d_sched_scratch,
                                        (unsigned*)(c->d_sched_scratch + kMaxBlocks * sizeof(Cand))));
  }
  EB_LAUNCH_CHECK(c, "schedule");
  if (h_res) {
    EB_CUDA(c, cudaMemcpyAsync(h_res, d_res, sizeof(eb_sched_result), cudaMemcpyDeviceToHost, st));
    EB_CUDA(c, cudaStreamSynchronize(st));
  }
  return EB_OK;
}
