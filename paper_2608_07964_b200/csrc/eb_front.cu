// The front end of a whole step, eb_step: everything between the inputs and the expert pass in three launches (four for
// many tokens).
//
//   front_kernel  : per chunk of <= 32 tokens: routing (a warp per token) and the chunk's assignments per expert
//   sums_kernel   : many tokens only: sums of the chunk histograms per 32 chunks, which one block would take too long over
//   tables_kernel : one block: loads, schedule, group table, tile plan
//   scatter_kernel: per part of a chunk: ranks, positions, gather of the token rows; some blocks fill the tile list
//
// The stages called one by one (eb_route, eb_schedule, eb_permute, eb_expert_ffn_grouped) take eight to eleven
// launches for the same tables.  What bounds these kernels is not work but the chain of hand-overs between them, each
// a launch, a first trip to memory and a few block barriers (2-5 us), so the split here follows the dependences that
// need the whole GPU to be through: the counts of all tokens, then the positions of all rows.  The counts travel as
// chunk histograms, which also spares the routing its global atomics.
#include <algorithm>

#include "eb_dispatch.cuh"
#include "eb_route.cuh"
#include "eb_schedule.cuh"
#include "eb_tiles.cuh"

namespace {

template <int PL>
__global__ void __launch_bounds__(kChunkThreads, PL <= 2 ? 2 : 1)
front_kernel(ModelParams mp, BatchParams bp, uint32_t pool_mask, uint32_t route_mask, const float* __restrict__ logits,
             int32_t* __restrict__ topk_idx, float* __restrict__ topk_w, int32_t* __restrict__ chunk_hist) {
  __shared__ int s_hist[EB_MAX_E];
  const int c = blockIdx.x, j = mb_of_chunk(bp, c);
  const int t = bp.tok_off[j] + (c - bp.chunk_off[j]) * 32 + (threadIdx.x >> 5), lane = threadIdx.x & 31;   // a warp per token
  const bool routed = (route_mask >> j) & 1u, counted = routed || ((pool_mask >> j) & 1u);
  if (counted && t < bp.tok_off[j + 1]) {
    if (routed && lane * 32 < mp.E) touch_ahead(logits + (size_t)t * mp.E + lane * 32);
    if (lane == 8) touch_ahead(topk_idx + (size_t)t * mp.K);
    if (routed && lane == 9) touch_ahead(topk_w + (size_t)t * mp.K);
  }
  EB_GRID_DEP_SYNC();
  if (!counted) return;
  route_chunk<PL>(mp, bp, c, j, routed, logits, topk_idx, topk_w, s_hist);
  for (int e = threadIdx.x; e < mp.E; e += kChunkThreads) chunk_hist[(size_t)c * mp.E + e] = s_hist[e];
}

// Running sum of n values that lie `stride` apart, left before each in `base` if `keep`; returns the total.  Sixteen loads at
// a time.
__device__ __forceinline__ int sum_chunks(const int32_t* __restrict__ h, int32_t* __restrict__ base, int n, int stride, bool keep) {
  int run = 0;
  for (int k0 = 0; k0 < n; k0 += 16) {
    int v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = k0 + k < n ? h[(size_t)(k0 + k) * stride] : 0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      if (keep && k0 + k < n) base[(size_t)(k0 + k) * stride] = run;
      run += v[k];
    }
  }
  return run;
}

// ---- sums ------------------------------------------------------------------------------------
// Segments of at most EB_SEG_CHUNKS chunks of one micro-batch.
struct Segments {
  int off[EB_MAX_MB + 1];   // first segment of every micro-batch; beyond n_mb: the total
};

// A thread per (segment, expert): chunk_base = assignments before the chunk in its segment, chunk_seg = of the segment.
// Only for steps whose histograms are too much for the one block of tables_kernel to add up (see kSumsWords).
__global__ void __launch_bounds__(256)
sums_kernel(const __grid_constant__ ModelParams mp, const __grid_constant__ BatchParams bp, const __grid_constant__ Segments seg, uint32_t counted,
            const int32_t* __restrict__ chunk_hist, int32_t* __restrict__ chunk_base, int32_t* __restrict__ chunk_seg) {
  EB_GRID_DEP_SYNC();
  const int i = blockIdx.x * 256 + threadIdx.x, g = i / mp.E, e = i - g * mp.E;
  if (g >= seg.off[EB_MAX_MB]) return;
  int j = 0;
  while (seg.off[j + 1] <= g) ++j;
  if (!((counted >> j) & 1u)) return;
  const int c0 = bp.chunk_off[j] + (g - seg.off[j]) * EB_SEG_CHUNKS;
  chunk_seg[i] = sum_chunks(chunk_hist + (size_t)c0 * mp.E + e, chunk_base + (size_t)c0 * mp.E + e, min((int)EB_SEG_CHUNKS, bp.chunk_off[j + 1] - c0), mp.E, true);
}

// ---- tables ----------------------------------------------------------------------------------
// The distinct layers of a batch, ascending.
struct StepLayers {
  int n;
  int layer[EB_MAX_MB];
  int mbs[EB_MAX_MB];     // micro-batches at the layer, as bits
  int of_mb[EB_MAX_MB];   // index of every micro-batch's layer
};

struct TablesArgs {
  uint32_t pool_mask, route_mask;
  int m, policy;
  const int32_t *chunk_hist, *chunk_seg;   // chunk_seg: null without sums_kernel
  int32_t *chunk_base, *seg_base, *mb_base, *mb_load, *mb_cnt;
  Segments seg;
  StepLayers layers;
  eb_sched_result* res;
  int32_t *group_off, *group_w, *step_meta;
  TilePlan plan;
  SchedGrid sched;
};

// i / E for i < 2^16 (E <= 256): one multiplication by ceil(2^32 / E); larger i take the division
__device__ __forceinline__ int div_by(int i, int E, unsigned magic) { return i < 65536 ? (int)__umulhi((unsigned)i, magic) : i / E; }

// One block, or several that all work out the loads, share the subsets of a MaxUtil schedule among them and leave the rest to
// the last one to arrive.  What bounds this kernel is its own chain of phases, a few hundred cycles each at best, a fifth of it
// waiting for instructions: every phase has a thread per item of the widest kind ((micro-batch, expert) or (layer, expert)), takes
// what it needs from shared memory, and decodes nothing by loops or divisions that a table or a multiplication gives; what does not
// depend on this step's routing is laid out while the kernel before still runs, the scans over groups and the order of the
// tiles share their barriers.  kLarge: a schedule of a large_pool; the others and the linear policies have a kernel without that code:
// steps of 4 x 64 tokens 31.85 -> 31.77 us, of 8 x 16 31.4 -> 31.0, under CumUtil 31.9 -> 31.3 and 33.5 -> 32.3, 5 x 93 tokens of odd
// sizes under DiffPeak 113.0 -> 110.8.  With one kernel for all and that code out of line, large pools took 0.5 us more.
template <bool kLarge>
__global__ void __launch_bounds__(kSchedThreads)
tables_kernel(const __grid_constant__ ModelParams mp, const __grid_constant__ BatchParams bp, const __grid_constant__ TablesArgs a) {
  extern __shared__ int4 s_dyn4[];
  __shared__ int4 s_expert[EB_MAX_E];               // in (device, expert) order: expert, first of its device, experts of the device, device
  __shared__ int s_dev_off[EB_MAX_D + 1], s_e2d[EB_MAX_E];
  __shared__ int s_home[EB_MAX_MB][EB_MAX_D + 1];   // first local token of every home device, per micro-batch
  __shared__ int s_layer[EB_MAX_MB], s_layer_mbs[EB_MAX_MB], s_layer_of[EB_MAX_MB];   // a.layers
  __shared__ int s_act[EB_MAX_MB];                  // active layers, ascending
  __shared__ int s_mbs[EB_MAX_MB];                  // their chosen micro-batches, as bits
  __shared__ int s_rank[EB_MAX_MB];                 // rank of every micro-batch's layer among them, -1 if not chosen
  __shared__ int s_nl;
  __shared__ int s_warp[32];
  __shared__ OrderShared s_order;
  SchedShared& sc = *reinterpret_cast<SchedShared*>(s_dyn4);
  int* const s_cnt = reinterpret_cast<int*>(s_dyn4) + sizeof(SchedShared) / 4;   // [n_mb][E] assignments, then rows before
  int* const s_goff = s_cnt + bp.n_mb * mp.E;                                    // [G + 1] group sizes, then offsets
  const int g_cap = bp.n_mb * (mp.E + mp.D * mp.S);
  int* const s_ptiles = s_goff + g_cap + 1;                                      // [G] tiles and cost class of every position
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int E = mp.E, S = mp.S, D = mp.D, n_mb = bp.n_mb;
  const bool first_block = blockIdx.x == 0;
  const unsigned magic = (unsigned)(((1ULL << 32) + E - 1) / E);   // E = 1: wraps to 0, see div_e
  auto div_e = [&](int i) { return E == 1 ? i : div_by(i, E, magic); };

  // ---- what depends on the model and on the arguments alone, before the kernels before this one are through: the expert tables
  // are written once, by eb_create
  if (tid <= D) s_dev_off[tid] = mp.dev_off[tid];
  if (tid < E) {
    const int e = mp.dev_list[tid], d = mp.e2d[e], off = mp.dev_off[d];
    s_expert[tid] = make_int4(e, off, mp.dev_off[d + 1] - off, d);
    s_e2d[e] = d;
  }
  if (tid >= 256 && tid < 256 + EB_MAX_MB * 16) {
    const int j = (tid - 256) / 16, d = tid % 16;
    if (j < n_mb && d <= D) {
      const int T = bp.tok_off[j + 1] - bp.tok_off[j];
      s_home[j][d] = home_start(d, T, D);
      if (d == 15 && D == 16) s_home[j][16] = T;
    }
  }
  if (tid >= 512 && tid < 512 + EB_MAX_MB * EB_MAX_D) sc.load[(tid - 512) / EB_MAX_D][tid % EB_MAX_D] = 0;
  if (tid >= 768 && tid < 768 + EB_MAX_MB) {
    const int i = tid - 768;
    s_layer[i] = a.layers.layer[i];
    s_layer_mbs[i] = i < a.layers.n ? a.layers.mbs[i] : 0;
    s_layer_of[i] = a.layers.of_mb[i];
  }
  for (int i = tid; i < kClasses * 33; i += kSchedThreads) (&s_order.warp[0][0])[i] = 0;
  if (tid < kClasses) s_order.carry[tid] = 0;
  schedule_prepare(sc, a.pool_mask, a.m, a.policy);
  __syncthreads();
  EB_GRID_DEP_SYNC();

  // ---- assignments of every (micro-batch, expert): from the segments' sums, or from the chunk histograms, which also gives
  // chunk_base = those before the chunk in its micro-batch; loads of the micro-batches routed now
  const uint32_t counted = a.pool_mask | a.route_mask;
  int kept = 0;   // a load of a micro-batch that keeps its routing
  if (tid >= kSchedThreads - EB_MAX_MB * EB_MAX_D) {
    const int j = (tid - (kSchedThreads - EB_MAX_MB * EB_MAX_D)) / EB_MAX_D, d = tid % EB_MAX_D;
    if (j < n_mb && d < D && !((a.route_mask >> j) & 1u)) sc.load[j][d] = kept = a.mb_load[j * D + d];
  }
  for (int i = tid; i < n_mb * E; i += kSchedThreads) {
    const int j = div_e(i), e = i - j * E;
    int n = 0;
    if ((counted >> j) & 1u) {
      if (a.chunk_seg) {
        const size_t at = (size_t)a.seg.off[j] * E + e;
        n = sum_chunks(a.chunk_seg + at, a.seg_base + at, a.seg.off[j + 1] - a.seg.off[j], E, first_block);
      } else {
        const size_t at = (size_t)bp.chunk_off[j] * E + e;
        n = sum_chunks(a.chunk_hist + at, a.chunk_base + at, bp.chunk_off[j + 1] - bp.chunk_off[j], E, first_block);
      }
    }
    s_cnt[i] = n;
    if ((a.route_mask >> j) & 1u) {
      if (first_block) a.mb_cnt[i] = n;
      if (n) atomicAdd(&sc.load[j][s_e2d[e]], n);
    }
  }
  // the loads of micro-batches routed now are at most their assignments
  const bool any_wide = __syncthreads_or(wide_load(kept)) || (long long)bp.n_tok * mp.K > kNarrowLoad;
  if (first_block && tid < EB_MAX_MB * EB_MAX_D) {
    const int j = tid / EB_MAX_D, d = tid % EB_MAX_D;
    if (j < n_mb && d < D && ((a.route_mask >> j) & 1u)) a.mb_load[j * D + d] = sc.load[j][d];
  }

  // ---- schedule; of several blocks the last one to arrive goes on
  uint32_t run;
  if (!schedule_grid<kLarge>(sc, D, a.pool_mask, a.m, a.policy, any_wide, a.sched, &run)) return;
  if (warp == 0) {
    // active layers: those with chosen micro-batches
    const int mbs = lane < EB_MAX_MB ? s_layer_mbs[lane] & (int)run : 0;
    const unsigned active = __ballot_sync(0xffffffffu, mbs != 0);
    if (mbs) {
      const int lr = __popc(active & ((1u << lane) - 1u));
      s_act[lr] = s_layer[lane];
      s_mbs[lr] = mbs;
    }
    if (lane < EB_MAX_MB) s_rank[lane] = (run >> lane) & 1u ? __popc(active & ((1u << s_layer_of[lane]) - 1u)) : -1;
    if (lane == 0) s_nl = __popc(active);
  }
  if (warp == 1) write_schedule(sc, D, a.pool_mask, run, a.res);
  __syncthreads();
  const int nl = s_nl, G = nl * (E + D * S);

  // ---- routed groups: sizes, weight matrices, tiles; s_cnt turns into the rows of a group before the micro-batch
  for (int i = tid; i < nl * E; i += kSchedThreads) {
    const int lr = div_e(i), k = i - lr * E;   // k: expert in (device, expert) order
    const int4 x = s_expert[k];
    const int e = x.x, off = x.y, n_d = x.z, d = x.w;
    int tot = 0;
    for (unsigned mbs = s_mbs[lr]; mbs; mbs &= mbs - 1) {
      int* at = s_cnt + (__ffs(mbs) - 1) * E + e;
      const int v = *at;
      *at = tot;
      tot += v;
    }
    const int g = nl * (off + d * S) + lr * (n_d + S) + (k - off);
    s_goff[g] = tot;
    a.group_w[g] = s_act[lr] * (E + S) + e;
    const int pos = nl * off + lr * n_d + (k - off), tiles = group_tiles(tot);
    s_ptiles[pos] = tiles << 4 | (cost_class(tiles, group_cols(tot)) & 15);
    a.plan.pgroup[pos] = g;
    a.plan.pslots[pos] = -1;
  }
  // ---- shared experts: rows = chosen tokens at the layer whose home device is d; the devices of a (layer, shared expert), as
  // positions neighbours, are sixteen neighbouring lanes
  for (int i0 = 0; i0 < nl * S * EB_MAX_D; i0 += kSchedThreads) {
    const int i = i0 + tid, q = i / EB_MAX_D, d = i % EB_MAX_D;
    const bool there = q < nl * S && d < D;
    const int lr = there ? q / S : 0, s = there ? q - lr * S : 0;
    int rows = 0;
    if (there)
      for (unsigned mbs = s_mbs[lr]; mbs; mbs &= mbs - 1) {
        const int j = __ffs(mbs) - 1;
        rows += s_home[j][d + 1] - s_home[j][d];
      }
    int n_slots = (rows + kSlotRows - 1) / kSlotRows, most = rows;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      n_slots += __shfl_xor_sync(0xffffffffu, n_slots, o);
      most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
    }
    if (!there) continue;
    const int off = s_dev_off[d], n_d = s_dev_off[d + 1] - off;
    const int g = nl * (off + d * S) + lr * (n_d + S) + n_d + s, pos = nl * E + q * D + d;
    s_goff[g] = rows;
    a.group_w[g] = s_act[lr] * (E + S) + E + s;
    const bool merged = D >= 2 && most <= kMergeMaxRows;
    const int tiles = !merged ? group_tiles(rows) : d == 0 ? (n_slots + kMergeSlots - 1) / kMergeSlots : 0;
    const int cols = merged ? merged_cols(min(n_slots, kMergeSlots)) : group_cols(rows);
    s_ptiles[pos] = tiles << 4 | (cost_class(tiles, cols) & 15);
    a.plan.pgroup[pos] = g;
    a.plan.pslots[pos] = merged ? n_slots : -1;
  }
  __syncthreads();

  // ---- exclusive scan over groups and order of the tiles of the expert pass, a chunk of 1024 groups and positions at a time (one
  // chunk as a rule)
  int carry = 0, my_cls = -1;
  long long my_at = 0;
  for (int b = 0; b < G; b += kSchedThreads) {
    const int i = b + tid;
    const int v = i < G ? s_goff[i] : 0, t = i < G ? s_ptiles[i] : 0;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += n;
    }
    if (lane == 31) s_warp[warp] = incl;
    my_cls = t >> 4 ? t & 15 : -1;
    my_at = order_mark(t >> 4, my_cls, s_order);
    __syncthreads();
    // every warp adds up the warps before it
    const int sum = s_warp[lane];
    const int excl = carry + (int)__reduce_add_sync(0xffffffffu, lane < warp ? sum : 0) + incl - v;
    carry += __reduce_add_sync(0xffffffffu, sum);
    if (i < G) {
      s_goff[i] = excl;
      a.group_off[i] = excl;
    }
    order_scan(s_order);
    __syncthreads();
    if (my_cls >= 0) my_at += s_order.warp[my_cls][warp];
    if (G > kSchedThreads) {
      if (i < G) order_park(i, my_cls, my_at, a.plan);
      __syncthreads();
      for (int k = tid; k < kClasses * 33; k += kSchedThreads) (&s_order.warp[0][0])[k] = 0;
      __syncthreads();
    }
  }
  if (G > kSchedThreads) {
    for (int i = tid; i < G; i += kSchedThreads) order_unpark(i, a.plan, s_order);
  } else {
    order_place(tid, my_cls, my_at, a.plan, s_order);
  }

  // ---- first row of every chosen (micro-batch, expert)
  for (int i = tid; i < n_mb * E; i += kSchedThreads) {
    const int j = div_e(i), k = i - j * E, lr = s_rank[j];
    if (lr < 0) continue;
    const int4 x = s_expert[k];
    const int at = j * E + x.x;
    a.mb_base[at] = s_cnt[at] + s_goff[nl * (x.y + x.w * S) + lr * (x.z + S) + (k - x.y)];
  }
  if (tid == 0) {
    a.group_off[G] = carry;
    a.step_meta[0] = carry;
    a.step_meta[1] = G;
    a.step_meta[2] = nl;
  }
  if (tid >= 32 && tid < 32 + EB_META_LEN - 3) {
    const int i = tid - 32;   // entries 3 .. EB_META_LEN-1
    a.step_meta[3 + i] = i < D ? nl * (s_dev_off[i] + i * S) : i == D ? G : 0;
  }
  if (tid == 64) order_finish(G, nl, -1, 0, a.plan, s_order);
}

// ---- scatter ---------------------------------------------------------------------------------
constexpr int kScatterThreads = 256;
constexpr int kScatterNarrow = 512;   // elements of a row up to which a block of many takes a whole chunk

struct ScatterArgs {
  const eb_sched_result* res;
  const int32_t *topk_idx, *chunk_base, *seg_base, *mb_base, *group_off, *group_w;   // seg_base: null without sums_kernel
  Segments seg;
  int32_t *pos, *row_src, *step_meta;
  const uint4* x;
  uint4* xp;
  TileList list;
  int fill_blocks;
  int team;   // threads per token row
  uint32_t touch_mask;   // micro-batches whose rows are asked for before it is known which run
  const int32_t* mb_load;
  ScheduleWatch watch;
};

// A watched schedule is copied to host memory by a block ahead of the others.  Blocks below fill_blocks write the tile list.  Each of the others places TB tokens of a chunk: the chunk's assignments up to
// them are ranked by warp matches while the token rows are on their way, then every row goes out to its K + S places, a team
// of threads per row.  What bounds it is that chain of two trips to memory and three barriers per block, and the row traffic.
// TB is small while there are few tokens (a block each keeps the chip busy) and 8 when there are many (ranking and tables are
// shared by more rows); one warp ranks.  Very many narrow rows take the whole chunk to a block: all warps rank, an assignment
// per thread, and the teams move several rows at once.  16 x 4096 tokens of 64 elements to 8 places took 109 us with one row at a
// time and TB = 8, 84 with teams and 29 with the whole chunk (44 for separate rank, gather and fill kernels), 16 x 2048 of 512
// elements 64 with teams and 46.  Wide rows need the blocks: with 2048 elements, 16 x 512 tokens take 45 us at TB = 8 and 74 at
// 32, with 1000 and 16 x 2048 both take 90.
template <int TB>
__global__ void __launch_bounds__(kScatterThreads)
scatter_kernel(const __grid_constant__ ModelParams mp, const __grid_constant__ BatchParams bp, const __grid_constant__ ScatterArgs a) {
  extern __shared__ int s_dyn[];
  int block = blockIdx.x;
  if (a.watch.rec && block-- == 0) {
    EB_GRID_DEP_SYNC();
    if (threadIdx.x < 32) leave_record(a.watch, a.res, a.mb_load, bp.n_mb * mp.D);
    return;
  }
  if (block < a.fill_blocks) {
    EB_GRID_DEP_SYNC();
    fill_tiles(mp, a.group_off, a.group_w, a.list, s_dyn, block, a.fill_blocks);
    return;
  }
  __shared__ StepShape ss;
  __shared__ int s_dev_off[EB_MAX_D + 1];
  __shared__ int s_next[EB_MAX_E];
  __shared__ int s_topk[32 * EB_MAX_K];
  constexpr bool kWide = TB == 32;
  __shared__ int s_count[kWide ? kScatterThreads / 32 : 1][EB_MAX_E];   // assignments of every expert in each warp
  __shared__ int s_pos[TB][EB_MAX_K + EB_MAX_S];
  static_assert(32 * EB_MAX_K <= kScatterThreads, "a thread per assignment of the chunk");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int E = mp.E, K = mp.K, S = mp.S, KS = K + S, vec = mp.H / 8;
  auto expert = [&](int e, int lane) { return (unsigned)e < (unsigned)E ? e : -1 - lane; };   // outside [0, E): equal to no other
  const int part = block - a.fill_blocks, c = part / (32 / TB);
  const int j = mb_of_chunk(bp, c);
  const int c0 = bp.tok_off[j] + (c - bp.chunk_off[j]) * 32;      // first token of the chunk
  const int t0 = c0 + part % (32 / TB) * TB;                      // and of this part
  const int nt = min(TB, bp.tok_off[j + 1] - t0);
  if (nt > 0 && ((a.touch_mask >> j) & 1u)) {
    // a line of 128 bytes per thread
    for (int i = tid * 8; i < nt * vec; i += kScatterThreads * 8) touch_ahead(a.x + (size_t)t0 * vec + i);
    if (tid * 32 < E) touch_ahead(a.mb_base + j * E + tid * 32);
    if (tid == 32) touch_ahead(a.topk_idx + (size_t)c0 * K);
  }
  EB_GRID_DEP_SYNC();
  if (nt <= 0) return;
  const uint32_t run = a.res->run_mask;
  if (!((run >> j) & 1u)) {
    for (int i = tid; i < nt * KS; i += kScatterThreads) a.pos[(size_t)t0 * KS + i] = -1;
    return;
  }
  // a team of threads per token row (one 16-byte column each); team 0 moves rows 0, teams, ..
  const int teams = kScatterThreads / a.team, team = tid / a.team, col0 = tid % a.team;
  // the first columns of the rows are on their way while the positions are worked out
  constexpr int P = TB < 8 ? TB : 8;   // rows in flight per thread
  uint4 v[P];
#pragma unroll
  for (int k = 0; k < P; ++k)
    if (team + k * teams < nt && col0 < vec) v[k] = __ldg(a.x + (size_t)(t0 + team + k * teams) * vec + col0);
  if (tid <= mp.D) s_dev_off[tid] = mp.dev_off[tid];
  // assignments from the start of the chunk to the end of this part
  const int first = (t0 - c0) * K, last = first + nt * K;
  if (tid < last) s_topk[tid] = a.topk_idx[(size_t)c0 * K + tid];
  if constexpr (kWide)
    for (int i = tid; i < E; i += kScatterThreads)
      for (int w = 0; w * 32 < last; ++w) s_count[w][i] = 0;
  const int32_t* seg_base = a.seg_base ? a.seg_base + (size_t)(a.seg.off[j] + (c - bp.chunk_off[j]) / EB_SEG_CHUNKS) * E : nullptr;
  for (int i = tid; i < E; i += kScatterThreads) s_next[i] = a.mb_base[j * E + i] + a.chunk_base[(size_t)c * E + i] + (seg_base ? seg_base[i] : 0);
  step_shape_block(bp, run, &ss);   // ends with a barrier
  // an index outside [0, E) is never used: the slot gets no row and the step's meta data counts it
  auto place = [&](int i, int p) {   // assignment i of the chunk, of this part
    const int t = c0 + i / K, k = i % K;
    a.pos[(size_t)t * KS + k] = p;
    s_pos[t - t0][k] = p;
    if (p >= 0) a.row_src[p] = t;
    else atomicAdd(&a.step_meta[EB_META_LEN - 1], 1);
  };
  const int ranker = kWide ? kScatterThreads / 32 - 1 : 0;   // the warp that also places the shared slots
  if constexpr (kWide) {
    // routed slots, a thread per assignment: the equal ones before it in its warp by a warp match, those of the warps before
    // it from the counts that each warp leaves
    const int e = tid < last ? expert(s_topk[tid], lane) : -1 - lane;
    const unsigned peers = __match_any_sync(0xffffffffu, e);
    const int before = __popc(peers & ((1u << lane) - 1u));
    if (e >= 0 && before == 0) s_count[warp][e] = __popc(peers);
    __syncthreads();
    if (tid < last) {
      int p = -1;
      if (e >= 0) {
        p = s_next[e] + before;
        for (int w = 0; w < warp; ++w) p += s_count[w][e];
      }
      place(tid, p);
    }
  } else if (warp == 0) {
    // routed slots in assignment order from the start of the chunk; the rows of the tokens before this part only count
    for (int a0 = 0; a0 < last; a0 += 32) {
      const int i = a0 + lane, e = i < last ? expert(s_topk[i], lane) : -1 - lane;
      const unsigned peers = __match_any_sync(0xffffffffu, e);
      const int before = __popc(peers & ((1u << lane) - 1u));
      if (i >= first && i < last) place(i, e >= 0 ? s_next[e] + before : -1);
      __syncwarp();
      if (e >= 0 && before == 0) s_next[e] += __popc(peers);
      __syncwarp();
    }
  }
  // shared slots: closed-form rows
  if (S > 0 && warp == ranker && lane < nt) {
    const int lr = ss.rank_of_mb[j], T = bp.tok_off[j + 1] - bp.tok_off[j], tl = t0 + lane - bp.tok_off[j];
    const int d = home_device(tl, T, mp.D);
    int before = 0;
    for (int j2 = 0; j2 < j; ++j2)
      if (ss.rank_of_mb[j2] == lr) {
        const int T2 = bp.tok_off[j2 + 1] - bp.tok_off[j2];
        before += home_start(d + 1, T2, mp.D) - home_start(d, T2, mp.D);
      }
    const int n_d = s_dev_off[d + 1] - s_dev_off[d];
    const int g = group_id(s_dev_off, S, ss.nl, d, lr, n_d), at = before + (tl - home_start(d, T, mp.D));
    for (int s = 0; s < S; ++s) {
      const int p = a.group_off[g + s] + at;
      a.pos[(size_t)(t0 + lane) * KS + K + s] = p;
      a.row_src[p] = t0 + lane;
      s_pos[lane][K + s] = p;
    }
  }
  __syncthreads();
  auto move_rows = [&](int row0, bool loaded) {
    for (int col = col0; col < vec; col += a.team) {
      if (!loaded) {
#pragma unroll
        for (int k = 0; k < P; ++k)
          if (row0 + k * teams < nt) v[k] = __ldg(a.x + (size_t)(t0 + row0 + k * teams) * vec + col);
      }
      loaded = false;
#pragma unroll
      for (int k = 0; k < P; ++k)
        if (row0 + k * teams < nt)
          for (int s = 0; s < KS; ++s) {
            const int p = s_pos[row0 + k * teams][s];
            if (p >= 0) a.xp[(size_t)p * vec + col] = v[k];
          }
    }
  };
  move_rows(team, true);
  if constexpr (TB > P)
    for (int row0 = team + P * teams; row0 < nt; row0 += P * teams) move_rows(row0, false);
}

// tables_kernel adds the chunk histograms up itself below this many words (chunks times experts) and up to this many chunks
// of one micro-batch: one block reads and writes them at the rate of one SM, and a thread per (micro-batch, expert) goes through
// a micro-batch's chunks in turn.  A launch of sums_kernel costs 2-3 us.  Steps without / with it (us, H = I = 64): 64 experts,
// 16 x 1024 tokens (32768 words) 128.1 / 131.2, 16 x 2048 225.2 / 223.9, 16 x 4096 400 / 389; 256 experts, 16 x 512 (65536)
// 117.0 / 118.3, 16 x 1024 190 / 183, 16 x 4096 616 / 559; 8 experts, 1 x 2048 (64 chunks) 42.4 / 42.0, 1 x 4096 50.3 / 46.0,
// 1 x 65536 346 / 193.
constexpr int kSumsWords = 65536;
constexpr int kSumsChunks = 64;

// tables_kernel runs on several blocks when the others take at least this many subsets of a MaxUtil schedule off the first:
// below, meeting in memory (0.6 to 1.4 us) costs more than it saves.  Steps on one / several blocks (us, 16 x 1 tokens, 64 experts):
// pool of 16 (eight blocks), m = 11 (6885 subsets) 33.5 / 32.2, m = 8 (39203) 46.2 / 32.5, m = 1 (65535) 56.6 / 33.0; pool of 15
// (four), m = 10 (4944) 31.2 / 31.9, m = 9 (9949) 32.7 / 31.7; pool of 14 (two), m = 8 (6476) 30.6 / 31.2, m = 6 (12911) 32.5 /
// 31.4.  256 experts: pool of 16, m = 1 62.8 / 39.0, m = 11 40.1 / 38.0; pool of 15, m = 10 37.8 / 37.9; pool of 14, m = 8 37.3 / 38.4.
constexpr int kSchedSubsets = 5000;

constexpr size_t tables_smem(int n_mb, int E, int groups) {
  return sizeof(SchedShared) + sizeof(int) * ((size_t)n_mb * E + 2 * (size_t)groups + 1);
}
// The most any shape takes.  The limit belongs to the kernel on its device: a context that set its own need would lower it for
// the contexts of larger shapes.
constexpr size_t kTablesSmemMax = tables_smem(EB_MAX_MB, EB_MAX_E, EB_MAX_MB * (EB_MAX_E + EB_MAX_D * EB_MAX_S));
static_assert(kTablesSmemMax + 16384 <= 232448, "shared memory of one block, the static part within 16 KB");

StepLayers layers_of(const BatchParams& bp) {
  StepLayers l = {};
  for (int j = 0; j < bp.n_mb; ++j) {
    int i = 0;
    while (i < l.n && l.layer[i] < bp.layer[j]) ++i;
    if (i == l.n || l.layer[i] != bp.layer[j]) {
      for (int k = l.n++; k > i; --k) {
        l.layer[k] = l.layer[k - 1];
        l.mbs[k] = l.mbs[k - 1];
      }
      l.layer[i] = bp.layer[j];
      l.mbs[i] = 0;
    }
    l.mbs[i] |= 1 << j;
  }
  for (int i = 0; i < l.n; ++i)
    for (int j = 0; j < bp.n_mb; ++j)
      if ((l.mbs[i] >> j) & 1) l.of_mb[j] = i;
  return l;
}

// Threads that move a row of `vec` 16-byte columns: the power of two that covers them, 8 to the whole block.
int row_team(int vec) {
  int t = 8;
  while (t < vec && t < kScatterThreads) t *= 2;
  return t;
}

}  // namespace

eb_status ebi_front_run(eb_ctx* c, cudaStream_t st, const BatchParams& bp, uint32_t pool_mask, uint32_t route_mask, int32_t m,
                        eb_policy policy, const eb_step_buffers* b) {
  const eb_config& g = c->cfg;
  if (!c->tables_attr_set) {   // per context: a context is on one device
    EB_CUDA(c, cudaFuncSetAttribute(tables_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTablesSmemMax));
    EB_CUDA(c, cudaFuncSetAttribute(tables_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTablesSmemMax));
    c->tables_attr_set = true;
  }
  if (bp.n_chunks > 0) {
    KernelTimer timer(c, EBK_ROUTE, st);
    EB_LAUNCH(c, "front", ebi_launch(g.E <= 64 ? front_kernel<2> : front_kernel<kMaxPerLane>, dim3(bp.n_chunks), dim3(kChunkThreads), 0, st, c->mp, bp,
                                     pool_mask, route_mask, (const float*)b->logits, b->topk_idx, b->topk_w, c->chunk_hist));
  }
  Segments seg;
  seg.off[0] = 0;
  for (int j = 0; j < EB_MAX_MB; ++j) seg.off[j + 1] = seg.off[j] + (bp.chunk_off[j + 1] - bp.chunk_off[j] + EB_SEG_CHUNKS - 1) / EB_SEG_CHUNKS;
  int longest = 0;
  for (int j = 0; j < bp.n_mb; ++j) longest = std::max(longest, bp.chunk_off[j + 1] - bp.chunk_off[j]);
  const bool sums = (int64_t)bp.n_chunks * g.E >= kSumsWords || longest > kSumsChunks;
  {
    KernelTimer timer(c, EBK_SCHEDULE, st);
    if (sums)
      EB_LAUNCH(c, "sums", ebi_launch(sums_kernel, dim3((seg.off[EB_MAX_MB] * g.E + 255) / 256), dim3(256), 0, st, c->mp, bp, seg, pool_mask | route_mask,
                                      (const int32_t*)c->chunk_hist, c->chunk_base, c->chunk_seg));
    const TablesArgs a{pool_mask, route_mask, (int)m, (int)policy, c->chunk_hist, sums ? c->chunk_seg : nullptr, c->chunk_base, c->seg_base,
                       c->mb_base, b->mb_load, b->mb_cnt, seg, layers_of(bp), b->sched, b->group_off, b->group_w, b->step_meta, tile_plan_of(c),
                       sched_grid_of(c)};
    int blocks = sched_blocks(pool_mask, m, policy);
    if ((int64_t)sched_subsets(pool_mask, m) * (blocks - 1) / blocks < kSchedSubsets) blocks = 1;
    const bool large = large_pool(__builtin_popcount(pool_mask), m, policy);
    EB_LAUNCH(c, "tables", ebi_launch(large ? tables_kernel<true> : tables_kernel<false>, dim3(blocks), dim3(kSchedThreads),
                                      tables_smem(bp.n_mb, g.E, bp.n_mb * (g.E + g.D * g.S)), st, c->mp, bp, a));
  }
  {
    KernelTimer timer(c, EBK_PERMUTE_GATHER, st);
    // Rows are asked for before the schedule says whether they are read: worth it if at least half of the pool is sure to run, and
    // never outside the pool.  Steps of 16 x 512 tokens (us, all rows / the pool's / by this rule): one of 2048 elements in the
    // pool 137.5 / 133.4 / 133.4, of 4096 74.6 / 72.5 / 72.5; all in the pool and m = 1 614 / 615 / 609 and 202.7 / 200.7 / 199.3,
    // m = 7 of 512 elements 101.3 / 100.0 / 98.1.  8 x 32 tokens of 2048, m = 6, 909.7 with and 908.3 either way.
    const int members = __builtin_popcount(pool_mask), sure = policy == EB_POLICY_ALL ? members : std::min((int)m, members);
    const uint32_t touch_mask = 2 * sure >= members ? pool_mask : 0;
    const ScatterArgs a{b->sched, b->topk_idx, c->chunk_base, sums ? c->seg_base : nullptr, c->mb_base, b->group_off, b->group_w, seg, b->pos, b->row_src, b->step_meta,
                        (const uint4*)b->x, (uint4*)b->xp, tile_list_of(c), c->num_sms / 2, row_team(g.H / 8), touch_mask,
                        b->mb_load, schedule_watch_of(c)};
    const size_t smem = sizeof(int) * (size_t)(ebi_groups_cap(c) + 1);
    auto launch = [&](auto kernel, int tb) {
      return ebi_launch(kernel, dim3((a.watch.rec ? 1 : 0) + a.fill_blocks + bp.n_chunks * (32 / tb)), dim3(kScatterThreads), smem, st, c->mp, bp, a);
    };
    EB_LAUNCH(c, "scatter", bp.n_tok <= 2 * c->num_sms     ? launch(scatter_kernel<1>, 1)
                            : bp.n_tok <= 16 * c->num_sms  ? launch(scatter_kernel<4>, 4)
                            : g.H > kScatterNarrow || bp.n_tok <= 64 * c->num_sms ? launch(scatter_kernel<8>, 8)
                                                                                  : launch(scatter_kernel<32>, 32));
  }
  ebi_watch_launched(c, st);
  EB_LAUNCH_CHECK(c, "step front end");
  return EB_OK;
}
