// eb_schedule: Schedule(S, m) of Algorithm 1 (eb_schedule.cuh) as a kernel of its own, one thread block, or several
// for MaxUtil over a large pool.
#include "eb_schedule.cuh"

namespace {

__global__ void __launch_bounds__(kSchedThreads)
schedule_kernel(int D, int n_mb, uint32_t pool_mask, int m, int policy, const int32_t* __restrict__ mb_load,
                eb_sched_result* __restrict__ res, SchedGrid grid) {
  EB_GRID_DEP_SYNC();
  __shared__ SchedShared s;
  const int tid = threadIdx.x;
  int load = 0;
  if (tid < EB_MAX_MB * EB_MAX_D) {
    const int j = tid / EB_MAX_D, d = tid % EB_MAX_D;
    if (j < n_mb && d < D) load = mb_load[j * D + d];
    s.load[j][d] = load;
  }
  schedule_prepare(s, pool_mask, m, policy);
  const bool any_wide = __syncthreads_or(wide_load(load));
  uint32_t run;
  if (!schedule_grid(s, D, pool_mask, m, policy, any_wide, grid, &run)) return;
  if (tid < 32) write_schedule(s, D, pool_mask, run, res);
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
    KernelTimer timer(c, EBK_SCHEDULE, st);
    EB_LAUNCH(c, "schedule", ebi_launch(schedule_kernel, dim3(sched_blocks(batch->pool_mask, m, policy)), dim3(kSchedThreads), 0, st, c->cfg.D,
                                        bp.n_mb, batch->pool_mask, (int)m, (int)policy, mb_load, d_res, sched_grid_of(c)));
  }
  EB_LAUNCH_CHECK(c, "schedule");
  if (h_res) {
    EB_CUDA(c, cudaMemcpyAsync(h_res, d_res, sizeof(eb_sched_result), cudaMemcpyDeviceToHost, st));
    EB_CUDA(c, cudaStreamSynchronize(st));
  }
  return EB_OK;
}
