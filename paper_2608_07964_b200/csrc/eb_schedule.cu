// eb_schedule: Schedule(S, m) of Algorithm 1 (eb_schedule.cuh) as a kernel of its own, one thread block, or several
// for MaxUtil over a large pool.
#include <cstring>

#include "eb_schedule.cuh"

namespace {

__global__ void __launch_bounds__(kSchedThreads)
schedule_kernel(int D, int n_mb, uint32_t pool_mask, int m, int policy, const int32_t* __restrict__ mb_load,
                eb_sched_result* res, SchedGrid grid, ScheduleWatch watch) {
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
  if (!schedule_grid<true>(s, D, pool_mask, m, policy, any_wide, grid, &run)) return;
  if (tid < 32) {
    write_schedule(s, D, pool_mask, run, res);
    if (watch.rec) {
      __syncwarp();
      leave_record(watch, res, mb_load, n_mb * D);
    }
  }
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
                                        bp.n_mb, batch->pool_mask, (int)m, (int)policy, mb_load, d_res, sched_grid_of(c), schedule_watch_of(c)));
    ebi_watch_launched(c, st);
  }
  EB_LAUNCH_CHECK(c, "schedule");
  if (h_res) {
    EB_CUDA(c, cudaMemcpyAsync(h_res, d_res, sizeof(eb_sched_result), cudaMemcpyDeviceToHost, st));
    EB_CUDA(c, cudaStreamSynchronize(st));
  }
  return EB_OK;
}

// Algorithm-1 loops wait for a schedule at every step.  Two blocking copies (result, loads) took 59 us of a scheduling step
// together with the kernels (eb_route's two and eb_schedule's), the record that the kernel leaves in host memory 30.
extern "C" eb_status eb_watch_schedule(eb_ctx* c, uint32_t ticket) {
  if (!c) return EB_ERR_INVALID_ARG;
  if (eb_status ds = ebi_check_device(c)) return ds;
  if (ticket && !c->watch_rec) {
    void* p = nullptr;
    EB_CUDA(c, cudaHostAlloc(&p, sizeof(ScheduleRecord), cudaHostAllocMapped | cudaHostAllocPortable));
    c->watch_rec = (ScheduleRecord*)p;
  }
  if (ticket) {
    __atomic_store_n(&c->watch_rec->ticket, 0u, __ATOMIC_RELEASE);
    c->watch_newest = ticket;
    c->watch_sent = 0;
  }
  c->watch_ticket = ticket;
  return EB_OK;
}

extern "C" eb_status eb_schedule_wait(eb_ctx* c, void* stream, uint32_t ticket, int32_t n_mb, const eb_sched_result* d_res, const int32_t* mb_load,
                                      eb_sched_result* h_res, int32_t* h_load) {
  if (!c) return EB_ERR_INVALID_ARG;
  if (!ticket || !d_res || !mb_load || !h_res) return ebi_fail(c, EB_ERR_INVALID_ARG, "null pointer or ticket 0");
  if (n_mb < 0 || n_mb > EB_MAX_MB) return ebi_fail(c, EB_ERR_UNSUPPORTED, "n_mb out of range");
  if (!c->watch_rec) return ebi_fail(c, EB_ERR_INVALID_ARG, "no schedule is watched");
  if (ticket != c->watch_newest) return ebi_fail(c, EB_ERR_INVALID_ARG, "not the last ticket that was set: its record may be written over");
  if (eb_status ds = ebi_check_device(c)) return ds;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t load_bytes = sizeof(int32_t) * (size_t)n_mb * c->cfg.D;
  auto marked = [&] { return __atomic_load_n(&c->watch_rec->ticket, __ATOMIC_ACQUIRE) == ticket; };
  for (unsigned spin = 1; !marked(); ++spin) {
    if (spin % 4096) continue;   // some microseconds between two questions to the runtime
    const cudaError_t e = cudaStreamQuery(st);
    if (e == cudaErrorNotReady) {
      cudaGetLastError();
      continue;
    }
    EB_CUDA(c, e);
    if (marked()) break;
    if (c->watch_sent == ticket) continue;   // launched on another stream than this one: the mark comes
    // everything enqueued here is over without a mark: a graph captured while nothing was watched
    EB_CUDA(c, cudaMemcpyAsync(h_res, d_res, sizeof(eb_sched_result), cudaMemcpyDeviceToHost, st));
    if (h_load) EB_CUDA(c, cudaMemcpyAsync(h_load, mb_load, load_bytes, cudaMemcpyDeviceToHost, st));
    EB_CUDA(c, cudaStreamSynchronize(st));
    return EB_OK;
  }
  *h_res = c->watch_rec->res;
  if (h_load) memcpy(h_load, c->watch_rec->load, load_bytes);
  return EB_OK;
}
