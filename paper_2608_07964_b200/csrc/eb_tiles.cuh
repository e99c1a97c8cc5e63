// The tile list of the expert pass: how groups are cut into tiles and in which order the tiles are dealt out.
#pragma once

#include "eb_internal.cuh"

namespace {

constexpr int kTileRows = 256;                                 // token rows of a tile at most
constexpr int kFeat1 = 256;                                    // outputs of a gate/up tile
constexpr int kFeat2 = 512;                                    // outputs of a down tile
constexpr int kSlotRows = 16;                                  // rows of one slot of a merged tile
constexpr int kMergeSlots = kTileRows / kSlotRows;             // slots of a merged tile at most
constexpr int kMergeMaxRows = 64;                              // replicas of a shared expert are merged when none has more rows

// Accumulator columns of a tile of `valid_rows` token rows: rounded up to 16 (each CTA of the pair supplies half
// of them, whole 8-row groups of the swizzled layout).
__device__ __forceinline__ int tile_cols(int valid_rows) {
  const int n = (valid_rows + 15) & ~15;
  return n > kTileRows ? kTileRows : n;
}
// Columns of a merged tile of n 16-row slots: an even number of slots, so that neither CTA's half cuts a slot.
__device__ __forceinline__ int merged_cols(int n_slots) { return ((n_slots + 1) & ~1) * kSlotRows; }
// Columns of a tile from its list entry (y = rows, or minus the slot count of a merged tile).
__device__ __forceinline__ int entry_cols(int y) { return y < 0 ? merged_cols(-y) : tile_cols(y); }

// One entry of the tile list.
struct Tile {
  int row;      // first row, or first slot of a merged tile
  int rows;     // rows (1 .. 256); -n for a merged tile of n slots of 16 rows, slots[row ..): (first row, rows)
  int w;        // weight matrix; negative: the list has ended
  int out;      // output tile
  int phase;    // 1: gate/up + SwiGLU (256 outputs per tile);  2: down (512 outputs per tile)
  int done;     // the token tile this one belongs to: entry of `ready`
  int need;     // phase 2: arrivals on that entry after which the rows of the intermediate are all written (0: they are)
  int once;     // no other token tile of the launch reads its matrix
};
static_assert(sizeof(Tile) == 32, "two 16-byte words");

// A group of `rows` rows is cut into ceil(rows / 256) tiles of nearly equal size, so no tile is a short
// remainder that would still stream a whole weight tile.
__device__ __forceinline__ int group_tiles(int rows) { return (rows + kTileRows - 1) / kTileRows; }
// Columns (token rows rounded up to 16) of the largest tile of a group; its cost class is that count in steps of 32.
__device__ __forceinline__ int group_cols(int rows) {
  const int t = group_tiles(rows);
  return t ? tile_cols((rows + t - 1) / t) : 0;
}

// Processing order of the groups.  The group table is device-major, so the D replicas of a shared
// expert (one group per virtual device, all reading the same weight matrix) lie far apart in it.
// Tiles are therefore listed in another order: first every routed group in table order, then the
// shared groups sorted by (layer, shared expert, device), so the replicas of one matrix are worked on
// side by side, share its tiles in L2 and the matrix leaves HBM once per step instead of D times.
// With a device filter (per-device timing) the device's own range is listed in table order.
__device__ __forceinline__ int group_at(const ModelParams& mp, const int* dev_off, int nl, int device, int g0, int i) {
  if (device >= 0) return g0 + i;
  const int routed = nl * mp.E;
  if (i < routed) {
    int d = 0;
    while (d + 1 < mp.D && i >= nl * dev_off[d + 1]) ++d;
    const int n_d = dev_off[d + 1] - dev_off[d];
    const int rel = i - nl * dev_off[d];
    return nl * (dev_off[d] + d * mp.S) + (rel / n_d) * (n_d + mp.S) + rel % n_d;
  }
  const int q = i - routed;
  const int lr = q / (mp.S * mp.D), s = (q / mp.D) % mp.S, d = q % mp.D;
  const int n_d = dev_off[d + 1] - dev_off[d];
  return nl * (dev_off[d] + d * mp.S) + lr * (n_d + mp.S) + n_d + s;
}

// The D replicas of a shared expert, when all are small, are packed into common tiles: the rows of each
// replica are cut into slots of 16 (one TMA box, one epilogue chunk), up to sixteen slots per tile, so the
// weight tile is fetched once for all of them.  `i` is a position of the processing order; returns true if
// it belongs to such a merged class and gives the class's first position and slot count.
__device__ __forceinline__ bool merged_class(const ModelParams& mp, const int* dev_off, int nl, int device, int i,
                                             const int32_t* __restrict__ group_off, int* head, int* n_slots) {
  if (device >= 0 || mp.S == 0 || mp.D < 2 || i < nl * mp.E) return false;
  const int q = i - nl * mp.E;
  const int h = i - q % mp.D;   // position of the class's replica on device 0
  int tot = 0, mx = 0;
  for (int d = 0; d < mp.D; ++d) {
    const int g = group_at(mp, dev_off, nl, device, 0, h + d);
    const int rows = group_off[g + 1] - group_off[g];
    tot += (rows + kSlotRows - 1) / kSlotRows;
    mx = rows > mx ? rows : mx;
  }
  *head = h;
  *n_slots = tot;
  return mx <= kMergeMaxRows;
}

// Cost classes of the tiles: class c holds the positions whose tiles have 32 c + 1 .. 32 (c + 1) columns.
constexpr int kClasses = kTileRows / 32;
__device__ __forceinline__ int cost_class(int tiles, int cols) { return tiles > 0 ? (cols + 31) / 32 - 1 : -1; }

struct TilePlan {
  int32_t *pgroup, *pslots;
  int4* prank;
  int32_t *order, *tile_pref, *work_count;
  int nt1, nt2;   // output tiles of the two phases
};
// One position of the processing order.
struct Position {
  int group, n_slots;   // n_slots: of its merged class, -1 otherwise
  int tiles, cls;       // tiles it owns (0: none, cls -1)
};
struct OrderShared {
  long long warp[kClasses][33];   // per class and warp: positions (low half) and tiles (high half), then those before the warp
  long long carry[kClasses];      // of the chunks of positions before
};

// The parts of order_tiles, which lists the positions that own tiles by cost class, widest tiles first, processing order inside
// a class, with the exclusive scan of their tile counts.  Widest-first order is what lets the expert kernel hand its tiles out to
// nearly equal ends.  Ranks inside a warp come from a warp match of the classes, the sums over warps from one warp per class: a
// block scan carrying all eight classes through every shuffle took three times as long.
//
// order_mark: a position per thread (class -1: none); returns the positions and tiles of its class in the lanes before it and
// leaves the warp's sums in sh.warp, which is clear.  Then a barrier, order_scan and another barrier.
__device__ __forceinline__ long long order_mark(int tiles, int cls, OrderShared& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned peers = __match_any_sync(0xffffffffu, cls), below = peers & ((1u << lane) - 1u);
  int pref = __popc(below);   // tiles of the class before this lane
  if (__any_sync(0xffffffffu, tiles > 1)) {
    unsigned todo = __ballot_sync(0xffffffffu, cls >= 0);
    while (todo) {
      const int c = __shfl_sync(0xffffffffu, cls, __ffs(todo) - 1);
      int incl = cls == c ? tiles : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
      }
      if (cls == c) pref = incl - tiles;
      todo &= ~__ballot_sync(0xffffffffu, cls == c);
    }
  }
  if (cls >= 0 && lane == 31 - __clz(peers))   // the class's last lane knows its sums
    sh.warp[cls][warp] = (long long)__popc(peers) | ((long long)(pref + tiles) << 32);
  return (long long)__popc(below) | ((long long)pref << 32);
}
// order_scan: sh.warp turns into those of the chunks and warps before, sh.carry takes the chunk up.
__device__ __forceinline__ void order_scan(OrderShared& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp >= kClasses) return;
  const long long v = sh.warp[warp][lane];
  long long incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long n = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += n;
  }
  const long long before = sh.carry[warp];
  sh.warp[warp][lane] = before + incl - v;
  __syncwarp();
  if (lane == 31) sh.carry[warp] = before + incl;
}
// order_place: position i of class cls, `at` of its class before it; sh.carry is final.
__device__ __forceinline__ void order_place(int i, int cls, long long at, const TilePlan& out, const OrderShared& sh) {
  if (cls < 0) return;
  for (int c = cls + 1; c < kClasses; ++c) at += sh.carry[c];   // the wider classes come first
  out.order[(int)(at & 0xffffffffLL)] = i;
  out.tile_pref[(int)(at & 0xffffffffLL)] = (int)(at >> 32);
}
// More than one chunk of positions: parked until the class bases are known (read back by the same thread).
__device__ __forceinline__ void order_park(int i, int cls, long long at, const TilePlan& out) {
  out.prank[i] = make_int4(cls, (int)(at & 0xffffffffLL), (int)(at >> 32), 0);
}
__device__ __forceinline__ void order_unpark(int i, const TilePlan& out, const OrderShared& sh) {
  const int4 v = out.prank[i];
  order_place(i, v.x, (long long)v.y | ((long long)v.z << 32), out, sh);
}
// The counts of the list; one thread.
__device__ __forceinline__ void order_finish(int ng, int nl, int device, int g0, const TilePlan& out, const OrderShared& sh) {
  long long all = 0;
  for (int c = 0; c < kClasses; ++c) all += sh.carry[c];
  const int n_listed = (int)(all & 0xffffffffLL), nt = (int)(all >> 32);
  out.tile_pref[n_listed] = nt;
  int32_t* const work_count = out.work_count;
  work_count[0] = nt * out.nt1;
  work_count[1] = nt * out.nt2;
  work_count[2] = nt;
  work_count[3] = g0;
  work_count[4] = ng;
  work_count[5] = n_listed;
  work_count[6] = work_count[7] = 0;   // tiles dealt out by the expert kernel
  work_count[8] = nl;
  work_count[9] = device;
}

// Orders the positions 0 .. ng - 1.  One block of 1024 threads; item(i) gives position i.
template <typename Item>
__device__ __forceinline__ void order_tiles(int ng, int nl, int device, int g0, Item item, const TilePlan& out, OrderShared& sh) {
  const int tid = threadIdx.x, warp = tid >> 5;
  int my_cls = -1;             // of the position this thread handled in the last chunk (the only one, as a rule)
  long long my_at = 0;
  if (tid < kClasses) sh.carry[tid] = 0;
  for (int b = 0; b < ng; b += 1024) {
    const int i = b + tid;
    Position p{0, -1, 0, -1};
    if (i < ng) {
      p = item(i);
      out.pgroup[i] = p.group;
      out.pslots[i] = p.n_slots;
    }
    if (tid < kClasses * 33) (&sh.warp[0][0])[tid] = 0;
    __syncthreads();
    my_at = order_mark(p.tiles, p.cls, sh);
    __syncthreads();
    order_scan(sh);
    __syncthreads();
    my_cls = p.cls;
    if (my_cls >= 0) my_at += sh.warp[my_cls][warp];
    if (ng > 1024) {
      if (i < ng) order_park(i, my_cls, my_at, out);
      __syncthreads();   // the table is cleared for the next chunk
    }
  }
  __syncthreads();
  if (ng > 1024) {
    for (int i = tid; i < ng; i += 1024) order_unpark(i, out, sh);
  } else {
    order_place(tid, my_cls, my_at, out, sh);
  }
  if (tid == 0) order_finish(ng, nl, device, g0, out, sh);
}

// fill: one thread per tile of the list (gate/up tiles, then down tiles); tiles of a group are ordered weight-tile
// major, token-tile minor.
// The function of block `block` of n_blocks.  s_pref: room for one int per group and one more; tile_pref is staged there
// once per block, the binary search below then stays on chip.
struct TileList {
  const int32_t *pgroup, *pslots, *order, *tile_pref, *work_count;
  int nt1, nt2, max_work;
  Tile* work;
  int32_t* ready;
  int2* slots;
};
__device__ __forceinline__ void fill_tiles(const ModelParams& mp, const int32_t* __restrict__ group_off, const int32_t* __restrict__ group_w,
                                           const TileList& l, int* s_pref, int block, int n_blocks) {
  const int32_t* __restrict__ pgroup = l.pgroup;
  const int32_t* __restrict__ pslots = l.pslots;
  const int32_t* __restrict__ order = l.order;
  const int32_t* __restrict__ tile_pref = l.tile_pref;
  const int nt1 = l.nt1, nt2 = l.nt2;
  int2* __restrict__ slots = l.slots;
  const int n_listed = l.work_count[5];
  const int cnt1 = l.work_count[0], total = cnt1 + l.work_count[1], nl = l.work_count[8], device = l.work_count[9];
  if (block * (int)blockDim.x >= total) return;
  for (int i = threadIdx.x; i <= n_listed; i += blockDim.x) s_pref[i] = tile_pref[i];
  __syncthreads();
  for (int idx = block * blockDim.x + threadIdx.x; idx < total; idx += n_blocks * blockDim.x) {
    const int list = idx >= cnt1 ? 1 : 0, local = idx - (list ? cnt1 : 0);
    const int nt = list ? nt2 : nt1;
    const int t_index = local / nt;
    // largest entry with tile_pref <= t_index (every listed position owns at least one tile)
    int lo = 0, hi = n_listed - 1;
    while (lo < hi) {
      int mid = (lo + hi + 1) >> 1;
      if (s_pref[mid] <= t_index) lo = mid; else hi = mid - 1;
    }
    const int t_g = s_pref[lo + 1] - s_pref[lo];
    const int rem = local - s_pref[lo] * nt;
    const int n = rem / t_g, m = rem % t_g;
    const int pos = order[lo], g = pgroup[pos], n_slots = pslots[pos];
    Tile it;
    if (n_slots >= 0) {
      // tile m of a merged class holds the next 16 slots of the class, replicas in device order
      const int base = kMergeSlots * (s_pref[lo] + m);
      const int first = kMergeSlots * m, n_here = min(kMergeSlots, n_slots - first);
      if (list == 0 && n == 0) {
        int c = 0;   // slots before the current replica
        for (int d = 0; d < mp.D; ++d) {
          const int gd = pgroup[pos + d];
          const int r0 = group_off[gd], rows = group_off[gd + 1] - r0;
          const int nc = (rows + kSlotRows - 1) / kSlotRows;
          for (int k = 0; k < nc; ++k, ++c)
            if (c >= first && c < first + n_here)
              slots[base + c - first] = make_int2(r0 + k * kSlotRows, min(kSlotRows, rows - k * kSlotRows));
        }
      }
      it.row = base;
      it.rows = -n_here;
    } else {
      // t_g tiles of nearly equal size: the first (rows % t_g) tiles hold one row more
      const int rows = group_off[g + 1] - group_off[g];
      const int each = rows / t_g, more = rows % t_g;
      it.row = group_off[g] + m * each + min(m, more);
      it.rows = each + (m < more ? 1 : 0);
    }
    it.w = group_w[g];
    it.out = n;
    it.phase = list + 1;
    it.done = s_pref[lo] + m;
    it.need = nt1 * 2;
    // the replicas of a shared expert that are not merged are tiles of their own over one matrix (with a device filter the
    // list holds one replica only)
    const bool replica = n_slots < 0 && device < 0 && mp.D > 1 && pos >= nl * mp.E;
    it.once = t_g == 1 && !replica;
    if (list == 0 && n == 0) l.ready[it.done] = 0;
    if (idx < l.max_work) l.work[idx] = it;
  }
}

// The context's tile tables as the planning and filling blocks take them.
inline TilePlan tile_plan_of(const eb_ctx* c) {
  const int nt1 = (c->cfg.I + kFeat1 - 1) / kFeat1, nt2 = (c->cfg.H + kFeat2 - 1) / kFeat2;
  return TilePlan{c->pgroup, c->pslots, c->prank, c->order, c->tile_pref, c->work_count, nt1, nt2};
}
inline TileList tile_list_of(const eb_ctx* c) {
  const TilePlan p = tile_plan_of(c);
  return TileList{c->pgroup, c->pslots, c->order, c->tile_pref, c->work_count, p.nt1, p.nt2, c->max_work, (Tile*)c->work, c->tile_ready, c->slots};
}

}  // namespace
