// Internal declarations shared by the translation units of libeb (not part of the ABI).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <string>
#include <vector>

#include "eb.h"

typedef __nv_bfloat16 bf16;

enum { EB_MAX_GUARDS = 24 };

// Chunks whose histograms one thread adds up in a whole step of many tokens.
enum { EB_SEG_CHUNKS = 32 };

// Kernel ids for the optional per-kernel event timing.
enum EbKernel {
  EBK_ROUTE = 0,
  EBK_SCHEDULE,
  EBK_PERMUTE_HIST,
  EBK_PERMUTE_SIZES,
  EBK_PERMUTE_SCAN,
  EBK_PERMUTE_RANK,
  EBK_PERMUTE_GATHER,
  EBK_FFN_PLAN,
  EBK_FFN_FILL,
  EBK_FFN_GATEUP,
  EBK_FFN_DOWN,
  EBK_COMBINE,
  EBK_PERMUTE_FUSED,
  EBK_COUNT
};

// Micro-batch description passed to kernels by value.
struct BatchParams {
  int32_t n_mb;
  int32_t n_tok;
  int32_t n_chunks;                 // chunks of <= 32 tokens, never straddling a micro-batch
  int32_t tok_off[EB_MAX_MB + 1];
  int32_t layer[EB_MAX_MB];
  int32_t chunk_off[EB_MAX_MB + 1]; // first chunk of every micro-batch
};

// Model description passed to kernels by value.
struct ModelParams {
  int32_t L, E, K, S, H, I, D, renorm;
  const int32_t* e2d;       // [E] expert -> device
  const int32_t* dev_off;   // [D+1] first entry of each device in dev_list
  const int32_t* dev_list;  // [E] routed experts sorted by (device, expert)
  const int32_t* e_local;   // [E] index of the expert among its device's experts
};

// Record of a schedule in pinned host memory (eb_watch_schedule).
struct ScheduleRecord {
  eb_sched_result res;
  int32_t load[EB_MAX_MB * EB_MAX_D];
  uint32_t ticket;   // written last
};
// Where a kernel leaves it: null: nowhere.
struct ScheduleWatch {
  ScheduleRecord* rec;
  uint32_t ticket;
};

struct eb_ctx {
  eb_config cfg;
  int device = 0;
  int num_sms = 0;
  std::vector<int32_t> e2d;
  int32_t* d_tables = nullptr;  // e2d | dev_off | dev_list | e_local
  ModelParams mp;
  int32_t* d_status = nullptr;
  ScheduleRecord* watch_rec = nullptr;   // pinned host memory, allocated on first use
  uint32_t watch_ticket = 0;
  uint32_t watch_newest = 0;             // last ticket set: the one that can be waited for
  uint32_t watch_sent = 0;               // ticket whose mark is sure to come: its kernels were launched, not captured
  char* d_sched_scratch = nullptr;  // per-block candidates and arrival counter of the multi-block scheduler

  const bf16* w_gate = nullptr;
  const bf16* w_up = nullptr;
  const bf16* w_down = nullptr;
  CUtensorMap tm_gate, tm_up, tm_down, tm_gate64, tm_up64;
  int pair_grid = 0;               // CTAs launched for the expert kernels: two per 2-CTA cluster the device holds at once

  // workspace carve-up
  void* ws = nullptr;
  size_t ws_bytes = 0;
  int n_guards = 0;                // guard areas between the regions below (debugging aid)
  size_t guard_off[EB_MAX_GUARDS] = {};
  int32_t* chunk_hist = nullptr;   // [max_chunks][E]
  int32_t* chunk_base = nullptr;   // [max_chunks][E]
  int32_t* chunk_seg = nullptr;    // [max_segs][E] assignments of every segment of chunks (whole steps of many tokens)
  int32_t* seg_base = nullptr;     // [max_segs][E] those before the segment in its micro-batch
  int32_t* mb_base = nullptr;      // [EB_MAX_MB][E] first row of every micro-batch in its groups (whole steps)
  int32_t* group_size = nullptr;   // [G_cap]
  int32_t* pgroup = nullptr;       // [G_cap] group at each position of the processing order
  int32_t* pslots = nullptr;       // [G_cap] 16-row slots of the merged shared-expert class of the position, -1 otherwise
  int4* prank = nullptr;           // [G_cap] (cost class, rank and tiles before it inside the class) when a plan has more than 1024 positions
  int32_t* order = nullptr;        // [G_cap] positions that own tiles, widest tiles first
  int32_t* tile_pref = nullptr;    // [G_cap + 1] tiles before each entry of `order`
  int32_t* work_count = nullptr;   // [16]: tile counts of the two phases, group range, dealt-out counters, layers, device filter
  void* work = nullptr;            // [max_work] tile list: gate/up tiles, then down tiles (32 bytes each)
  int32_t* tile_ready = nullptr;   // [max_tiles] per token tile: finished parts of its intermediate rows
  int2* slots = nullptr;           // [16 * max_tiles] (first row, rows) of the 16-row slots of merged tiles
  bf16* act = nullptr;             // [R_cap][I]
  int32_t max_chunks = 0, max_tiles = 0, max_work = 0;

  bool fused_attr_set = false, tables_attr_set = false;
  // eb_step_host_submit / eb_step_host_wait: copy streams and per-slot events, created on first use
  cudaStream_t s_in = nullptr, s_out = nullptr;
  cudaEvent_t ev_in[EB_HOST_SLOTS] = {}, ev_step[EB_HOST_SLOTS] = {}, ev_out[EB_HOST_SLOTS] = {};
  bool slot_busy[EB_HOST_SLOTS] = {};
  bool timing = false;
  cudaEvent_t ev[2 * EBK_COUNT] = {};
  bool ev_valid[EBK_COUNT] = {};

  std::string err;
};

// After the launch of the kernel that leaves the record: its mark comes, on whatever stream that was.  A captured launch promises nothing.
inline void ebi_watch_launched(eb_ctx* c, cudaStream_t st) {
  if (!c->watch_ticket) return;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) cudaGetLastError();
  else if (cap == cudaStreamCaptureStatusNone) c->watch_sent = c->watch_ticket;
}
inline ScheduleWatch schedule_watch_of(const eb_ctx* c) { return ScheduleWatch{c->watch_ticket ? c->watch_rec : nullptr, c->watch_ticket}; }

int32_t ebi_rows_cap(const eb_ctx* c);
int32_t ebi_groups_cap(const eb_ctx* c);
eb_status ebi_fail(eb_ctx* c, eb_status s, const std::string& msg);
eb_status ebi_check_cuda(eb_ctx* c, cudaError_t e, const char* what);
eb_status ebi_make_batch(eb_ctx* c, const eb_batch* b, BatchParams* out);
// EB_OK if the calling thread's current device is the one the context was created on.
eb_status ebi_check_device(eb_ctx* c);

// Brackets a launch with events when timing is enabled.
struct KernelTimer {
  eb_ctx* c;
  int id;
  cudaStream_t s;
  KernelTimer(eb_ctx* ctx, int kid, cudaStream_t st) : c(ctx), id(kid), s(st) {
    if (c->timing) cudaEventRecord(c->ev[2 * id], s);
  }
  ~KernelTimer() {
    if (c->timing) {
      cudaEventRecord(c->ev[2 * id + 1], s);
      c->ev_valid[id] = true;
    }
  }
};

#define EB_CUDA(ctx, expr)                                              \
  do {                                                                  \
    cudaError_t _e = (expr);                                            \
    if (_e != cudaSuccess) return ebi_check_cuda((ctx), _e, #expr);     \
  } while (0)

// A launch.  The kernels of a call work from what those before them wrote, so one that is refused ends the call.
#define EB_LAUNCH(ctx, what, expr)                                      \
  do {                                                                  \
    cudaError_t _e = (expr);                                            \
    if (_e != cudaSuccess) {                                            \
      cudaGetLastError();                                               \
      return ebi_check_cuda((ctx), _e, what);                           \
    }                                                                   \
  } while (0)

#define EB_LAUNCH_CHECK(ctx, what)                                      \
  do {                                                                  \
    cudaError_t _e = cudaGetLastError();                                \
    if (_e != cudaSuccess) return ebi_check_cuda((ctx), _e, what);      \
  } while (0)

// Every kernel of the library calls EB_GRID_DEP_SYNC() before it reads what a kernel may have written and before it writes: it waits
// until the kernels before it in the stream have finished (and their writes are visible), then lets the kernel after it start being
// scheduled.  Before it stand at most hints (touch_ahead) and, in tables_kernel, shared memory laid out from the arguments
// and from tables that eb_create wrote.  With launches made through ebi_launch (programmatic stream serialisation) the launch
// latency of each small kernel overlaps the previous kernel; with ordinary launches it is a no-op.
#define EB_GRID_DEP_SYNC() asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" ::: "memory")

// Asks for the line at `p` to be in L2, without waiting and without reading anything, so that it may stand before
// EB_GRID_DEP_SYNC().  Only for what the kernel is sure, or likely, to need: a line that nobody reads costs its transfer and another
// line's place.  A step streams more than L2 holds, so its inputs and tables are in HBM when the next one begins: routing
// 2.8 -> 2.1 us (8 x 32 tokens) and 6.6 -> 5.2 (16 x 512), scatter there 46 -> 42, aggregation 5.4 -> 4.6 (8 x 32).
__device__ __forceinline__ void touch_ahead(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Number of kernels this library has launched in the process (all contexts).
extern std::atomic<unsigned long long> g_ebi_launches;

template <typename... KArgs, typename... Args>
static inline cudaError_t ebi_launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                     Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  ++g_ebi_launches;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

static inline bool ebi_aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Entry points of the per-step stages (defined in their own translation units).
eb_status ebi_ffn_run(eb_ctx* c, cudaStream_t st, const void* xp, const int32_t* group_off,
                      const int32_t* group_w, const int32_t* step_meta, void* yp, int32_t device, bool planned = false);
// Routing, schedule, dispatch tables, gather and tile list of a whole step (eb_front.cu).
eb_status ebi_front_run(eb_ctx* c, cudaStream_t st, const BatchParams& bp, uint32_t pool_mask, uint32_t route_mask, int32_t m,
                        eb_policy policy, const eb_step_buffers* b);
eb_status ebi_ffn_bind(eb_ctx* c);
eb_status ebi_selftest_wait(eb_ctx* c, cudaStream_t st, long long limit_cycles, int* d_gave_up);
