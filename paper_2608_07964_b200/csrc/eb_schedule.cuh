// Schedule(S, m) of Algorithm 1 for one thread block: the policies and the result record.
//
// MaxUtil (Section 4.2) enumerates every subset of the pool with at least m members.  The pool
// is split into a low and a high half; the summed load vector of each half-subset is tabulated
// in shared memory (2 x 256 x D entries at most), so a subset costs D additions and a maximum.
// Utilisation (Eq. 3 for one step) is sum(W) / (D * max(W)); D is common to all candidates, so
// candidates are compared exactly by cross-multiplying sum and max in 64-bit integers.
// Total order: higher utilisation, then more members, then the numerically smaller mask.
// CumUtil / DiffPeak (Section 5.2) go through the pool in order, one warp with a device per lane; topping their result
// up to m members scores the remaining pool members in parallel, one lane each.
//
// What bounds the enumeration is instruction issue: 2^16 subsets on one SM.  Subsets that are too small are not visited:
// the low halves are kept in the order of their member counts, so that for every high half the sufficient ones come
// first (12 of 16 members: 212 warp turns instead of 2048).  Sums are 32-bit where the loads allow it, and the tables'
// rows are 20 words apart, which 16-byte reads of neighbouring rows go through without bank conflicts.
#pragma once

#include "eb_internal.cuh"

namespace {

constexpr int kSchedThreads = 1024;
constexpr int kSchedRow = EB_MAX_D + 4;   // words between rows of the subset tables
constexpr int kNarrowLoad = 1 << 22;      // loads up to here: every sum over micro-batches and devices fits 31 bits

struct Cand {
  long long num;   // sum_d W_d  (D if there is no work: U := 1)
  long long peak;  // max_d W_d  (1 if there is no work)
  int n;           // members
  unsigned sub;    // subset in pool-relative bit positions (order preserving w.r.t. the real mask)
};

__device__ __forceinline__ bool better(const Cand& a, const Cand& b) {
  if (b.n < 0) return a.n >= 0;
  if (a.n < 0) return false;
  long long l = a.num * b.peak, r = b.num * a.peak;
  if (l != r) return l > r;
  if (a.n != b.n) return a.n > b.n;
  return a.sub < b.sub;
}

// utilisation of a joint load whose entries lie in the lanes of a warp (zero beyond D)
__device__ __forceinline__ Cand warp_util(long long w, int D, bool wide) {
  Cand c;
  if (wide) {
    long long num = w, peak = w;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      num += __shfl_xor_sync(0xffffffffu, num, o);
      const long long p2 = __shfl_xor_sync(0xffffffffu, peak, o);
      peak = p2 > peak ? p2 : peak;
    }
    c.num = num;
    c.peak = peak;
  } else {
    c.num = __reduce_add_sync(0xffffffffu, (int)w);
    c.peak = __reduce_max_sync(0xffffffffu, (int)w);
  }
  if (c.peak == 0) {
    c.num = D;
    c.peak = 1;
  }
  c.n = 0;
  c.sub = 0;
  return c;
}

// best candidate of the warp, in every lane
__device__ __forceinline__ Cand warp_best(Cand c) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Cand oth;
    oth.num = __shfl_xor_sync(0xffffffffu, c.num, o);
    oth.peak = __shfl_xor_sync(0xffffffffu, c.peak, o);
    oth.n = __shfl_xor_sync(0xffffffffu, c.n, o);
    oth.sub = __shfl_xor_sync(0xffffffffu, c.sub, o);
    if (better(oth, c)) c = oth;
  }
  return c;
}
// the same for candidates whose numbers fit 32 bits and whose n is the member count of sub (or negative: none)
__device__ __forceinline__ Cand warp_best_narrow(const Cand& c0) {
  int num = (int)c0.num, peak = (int)c0.peak;
  unsigned sub = c0.n < 0 ? 0u : c0.sub;   // the empty subset is never a candidate
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int num2 = __shfl_xor_sync(0xffffffffu, num, o), peak2 = __shfl_xor_sync(0xffffffffu, peak, o);
    const unsigned sub2 = __shfl_xor_sync(0xffffffffu, sub, o);
    const long long l = (long long)num2 * peak, r = (long long)num * peak2;
    const int n = __popc(sub), n2 = __popc(sub2);
    if (n2 != 0 && (n == 0 || l > r || (l == r && (n2 > n || (n2 == n && sub2 < sub))))) {
      num = num2;
      peak = peak2;
      sub = sub2;
    }
  }
  Cand c;
  c.num = num;
  c.peak = peak;
  c.n = sub ? __popc(sub) : -1;
  c.sub = sub;
  return c;
}


// run set of a candidate; one warp
__device__ __forceinline__ uint32_t run_mask_of(const int* member, int np, const Cand& b) {
  const int k = threadIdx.x & 31;
  return __reduce_or_sync(0xffffffffu, k < np && ((b.sub >> k) & 1u) ? 1u << member[k] : 0u);
}

// The byte values, those with more bits set first, then ascending.
struct ByCount {
  alignas(4) unsigned char v[256];
};
constexpr ByCount make_by_count() {
  ByCount t{};
  int at = 0;
  for (int n = 8; n >= 0; --n)
    for (int u = 0; u < 256; ++u) {
      int bits = 0;
      for (int b = 0; b < 8; ++b) bits += (u >> b) & 1;
      if (bits == n) t.v[at++] = (unsigned char)u;
    }
  return t;
}
static __device__ const ByCount kByCount = make_by_count();

struct SchedShared {
  int4 lo[256 * kSchedRow / 4], hi[256 * kSchedRow / 4];   // summed loads of every subset of the two halves of the pool
  int load[EB_MAX_MB][EB_MAX_D];                           // zero beyond n_mb and D
  int nibble[4][16][EB_MAX_D];                             // summed loads of every subset of four pool positions
  unsigned char by_count[256];                             // kByCount
  int member[EB_MAX_MB];                                   // micro-batch of every pool position
  Cand best[kSchedThreads / 32];
  uint32_t run;
  bool last;                                               // this block is the last one of the grid to arrive
  long long seq_w[EB_MAX_D];
};

// Joint load of the low-half subset lo and a high-half one whose loads are in hi: compared with the best so far.
template <typename W>
struct BestSubset {
  W num = 0, peak = 1;
  int n = -1;
  unsigned sub = 0;
  __device__ __forceinline__ void offer(const int4* lo, const int4* hi, int quads, int D, int n2, unsigned sub2) {
    W num2 = 0, peak2 = 0;
    for (int q = 0; q < quads; ++q) {   // entries beyond D are zero
      const int4 a = lo[q], b = hi[q];
      const W w0 = (W)a.x + b.x, w1 = (W)a.y + b.y, w2 = (W)a.z + b.z, w3 = (W)a.w + b.w;
      num2 += (w0 + w1) + (w2 + w3);
      const W p0 = w0 > w1 ? w0 : w1, p1 = w2 > w3 ? w2 : w3, p = p0 > p1 ? p0 : p1;
      peak2 = p > peak2 ? p : peak2;
    }
    if (peak2 == 0) {
      num2 = D;
      peak2 = 1;
    }
    const long long l = (long long)num2 * peak, r = (long long)num * peak2;
    if (n < 0 || l > r || (l == r && (n2 > n || (n2 == n && sub2 < sub)))) {
      num = num2;
      peak = peak2;
      n = n2;
      sub = sub2;
    }
  }
};

// Best subset (pool positions as bits) of at least m members among this block's share.
template <typename W>
__device__ __forceinline__ Cand maxutil_scan(const SchedShared& s, int D, int np, int nlo, int m, int block, int n_blocks) {
  const int quads = (D + 3) / 4, tid = threadIdx.x;
  static_assert(EB_MAX_D == 16 && EB_MAX_MB == 16, "the tables are indexed in nibbles");
  BestSubset<W> best;
  if (np <= 10) {   // a subset per thread
    const int n = __popc(tid);
    if (tid < (1 << np) && n >= m)
      best.offer(s.lo + (tid & ((1 << nlo) - 1)) * (kSchedRow / 4), s.hi + (tid >> nlo) * (kSchedRow / 4), quads, D, n, tid);
  } else {
    // A warp takes high halves in turn and, for each, the low halves that bring it to m members: they come first in
    // the order by member count.  Which warp takes which high half changes from turn to turn, so that the shares of
    // large high halves even out.
    const int lane = tid & 31, warp = tid >> 5;
    for (int k = block; k < (1 << (np - 8)) / 32 + 1; k += n_blocks) {
      const int h = k * 32 + (warp ^ (k * 11 & 31)), n_h = __popc(h);
      if (h >= 1 << (np - 8)) continue;
      const int need = max(0, m - n_h);
      if (need > 8) continue;
      // byte values with at least `need` bits set: 256, 255, 247, 219, 163, 93, 37, 9, 1
      const int n_lo = need == 0 ? 256 : (int)((0x0109255da3dbf7ffULL >> (8 * (need - 1))) & 255u);
      const int4* hi = s.hi + h * (kSchedRow / 4);
      for (int i = lane; i < n_lo; i += 32) {
        const int u = s.by_count[i];
        if (u | h) best.offer(s.lo + u * (kSchedRow / 4), hi, quads, D, n_h + __popc(u), (unsigned)(h << 8 | u));
      }
    }
  }
  Cand c;
  c.num = best.num;
  c.peak = best.peak;
  c.n = best.n;
  c.sub = best.sub;
  return c;
}

// Chooses the run set from s.load.  All kSchedThreads threads of the block call it after a barrier behind the writes of
// s.load; `block` of n_blocks.  On return (after a barrier): s.run, or with n_blocks > 1 under MaxUtil this block's
// candidate in s.best[0].  True: s.run is final.
__device__ __forceinline__ bool schedule_block(SchedShared& s, int D, uint32_t pool_mask, int m, int policy, int block, int n_blocks) {
  const int tid = threadIdx.x;
  const int np = __popc(pool_mask);
  if (tid < EB_MAX_MB && ((pool_mask >> tid) & 1u)) s.member[__popc(pool_mask & ((1u << tid) - 1u))] = tid;
  if (np <= m || policy == EB_POLICY_ALL) {
    if (tid == 0) s.run = pool_mask;
    __syncthreads();
    return true;
  }
  bool wide = false;
  if (tid < EB_MAX_MB * EB_MAX_D) {
    const int v = s.load[tid / EB_MAX_D][tid % EB_MAX_D];
    wide = v < 0 || v > kNarrowLoad;
  }
  const bool any_wide = __syncthreads_or(wide);
  if (policy == EB_POLICY_MAXUTIL) {
    const int nlo = np < 8 ? np : 8, nhi = np - nlo;
    int* lo = reinterpret_cast<int*>(s.lo);
    int* hi = reinterpret_cast<int*>(s.hi);
    // sums over four members at a time (one entry per thread), then over eight
    {
      const int quad = tid >> 8, u = (tid >> 4) & 15, d = tid & 15;
      int acc = 0;
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (quad * 4 + b < np && ((u >> b) & 1)) acc += s.load[s.member[quad * 4 + b]][d];
      s.nibble[quad][u][d] = acc;
    }
    if (np > 10 && tid < 64) reinterpret_cast<uint32_t*>(s.by_count)[tid] = reinterpret_cast<const uint32_t*>(kByCount.v)[tid];
    __syncthreads();
    for (int i = tid; i < (1 << nlo) * EB_MAX_D; i += kSchedThreads)
      lo[(i >> 4) * kSchedRow + (i & 15)] = s.nibble[0][(i >> 4) & 15][i & 15] + s.nibble[1][i >> 8][i & 15];
    for (int i = tid; i < (1 << nhi) * EB_MAX_D; i += kSchedThreads)
      hi[(i >> 4) * kSchedRow + (i & 15)] = s.nibble[2][(i >> 4) & 15][i & 15] + s.nibble[3][i >> 8][i & 15];
    __syncthreads();
    Cand best = any_wide ? maxutil_scan<long long>(s, D, np, nlo, m, block, n_blocks) : maxutil_scan<int>(s, D, np, nlo, m, block, n_blocks);
    // warp then block reduction under the total order (any reduction order gives the same winner)
    best = any_wide ? warp_best(best) : warp_best_narrow(best);
    if ((tid & 31) == 0) s.best[tid >> 5] = best;
    __syncthreads();
    if (tid < 32) {
      Cand b = any_wide ? warp_best(s.best[tid]) : warp_best_narrow(s.best[tid]);
      const uint32_t mask = run_mask_of(s.member, np, b);
      if (tid == 0) {
        s.best[0] = b;
        s.run = mask;
      }
    }
    __syncthreads();
    return n_blocks == 1;
  }
  if (tid < 32) {
    // CumUtil / DiffPeak: ascending pool members, the first always taken; lane d holds the joint load of device d
    const int lane = tid;
    auto load_of = [&](int j) { return lane < EB_MAX_D ? (long long)s.load[j][lane] : 0LL; };
    long long w = load_of(s.member[0]);
    uint32_t run = 1u << s.member[0];
    int n = 1;
    if (policy == EB_POLICY_CUMUTIL) {
      Cand cur = warp_util(w, D, any_wide);
      for (int k = 1; k < np; ++k) {
        const int j = s.member[k];
        const long long w2 = w + load_of(j);
        const Cand nxt = warp_util(w2, D, any_wide);
        if (nxt.num * cur.peak > cur.num * nxt.peak) {
          w = w2;
          cur = nxt;
          run |= 1u << j;
          ++n;
        }
      }
    } else {
      int my_peak = 0;   // device with the largest load of pool member `lane`, the lowest index among equals
      if (lane < np)
        for (int d = 1; d < D; ++d)
          if (s.load[s.member[lane]][d] > s.load[s.member[lane]][my_peak]) my_peak = d;
      uint32_t peaks = 1u << __shfl_sync(0xffffffffu, my_peak, 0);
      for (int k = 1; k < np; ++k) {
        const uint32_t bit = 1u << __shfl_sync(0xffffffffu, my_peak, k);
        if (peaks & bit) continue;
        peaks |= bit;
        w += load_of(s.member[k]);
        run |= 1u << s.member[k];
        ++n;
      }
    }
    if (lane < EB_MAX_D) s.seq_w[lane] = w;
    __syncwarp();
    // top up to m members: repeatedly add the member whose inclusion gives the highest utilisation
    // (lowest index on ties); lane k scores pool member k
    while (n < m) {
      Cand cu;
      cu.n = -1; cu.num = 0; cu.peak = 1; cu.sub = 0;
      if (lane < np && !((run >> s.member[lane]) & 1u)) {
        long long num = 0, peak = 0;
#pragma unroll
        for (int d = 0; d < EB_MAX_D; ++d) {   // zero beyond D
          const long long v = s.seq_w[d] + s.load[s.member[lane]][d];
          num += v;
          peak = v > peak ? v : peak;
        }
        cu.num = peak ? num : D;
        cu.peak = peak ? peak : 1;
        cu.n = 1;                 // equal sizes: ties fall to the lower index
        cu.sub = (unsigned)lane;
      }
      cu = warp_best(cu);
      if (cu.n < 0) break;
      const int bj = s.member[cu.sub];
      __syncwarp();
      if (lane < EB_MAX_D) s.seq_w[lane] += s.load[bj][lane];
      __syncwarp();
      run |= 1u << bj;
      ++n;
    }
    if (lane == 0) s.run = run;
  }
  __syncthreads();
  return true;
}

// schedule_block by all blocks of the grid: each leaves its best candidate in global memory and the block that arrives last
// goes on with the choice among them.  False: this block is done.  The counter is ready for the next launch again.
struct SchedGrid {
  Cand* best;          // [gridDim.x]
  unsigned* arrived;
};
__device__ __forceinline__ bool schedule_grid(SchedShared& s, int D, uint32_t pool_mask, int m, int policy, const SchedGrid& g) {
  if (schedule_block(s, D, pool_mask, m, policy, blockIdx.x, gridDim.x)) return gridDim.x == 1 || blockIdx.x == 0;
  const int tid = threadIdx.x;
  if (tid == 0) {
    g.best[blockIdx.x] = s.best[0];
    __threadfence();
    s.last = atomicAdd(g.arrived, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s.last) return false;
  __threadfence();
  if (tid < 32) {
    Cand b;
    b.n = -1; b.num = 0; b.peak = 1; b.sub = 0;
    for (int i = tid; i < (int)gridDim.x; i += 32) {
      const Cand o = g.best[i];
      if (better(o, b)) b = o;
    }
    b = warp_best(b);
    const uint32_t mask = run_mask_of(s.member, __popc(pool_mask), b);
    if (tid == 0) {
      s.run = mask;
      *g.arrived = 0;
    }
  }
  __syncthreads();
  return true;
}

// Blocks for a schedule: MaxUtil over a pool of more than 13 takes one per 32 high halves of its subsets.
constexpr int kMaxSchedBlocks = 1 << (EB_MAX_MB - 13);
inline int sched_blocks(uint32_t pool_mask, int m, int policy) {
  const int np = __builtin_popcount(pool_mask);
  return policy == EB_POLICY_MAXUTIL && np > m && np > 13 ? 1 << (np - 13) : 1;
}
// Subsets that MaxUtil looks at: those of at least m members.
inline int sched_subsets(uint32_t pool_mask, int m) {
  const int np = __builtin_popcount(pool_mask);
  int total = 0, c = 1;   // c: n out of np
  for (int n = 0; n <= np; ++n) {
    if (n >= m) total += c;
    c = c * (np - n) / (n + 1);
  }
  return total;
}
inline SchedGrid sched_grid_of(const eb_ctx* c) {
  return SchedGrid{(Cand*)c->d_sched_scratch, (unsigned*)(c->d_sched_scratch + kMaxSchedBlocks * sizeof(Cand))};
}

// The result record, by one warp, s.run final.
__device__ __forceinline__ void write_schedule(const SchedShared& s, int D, uint32_t pool_mask, eb_sched_result* __restrict__ res) {
  const int tid = threadIdx.x & 31;
  // lane d sums the chosen micro-batches' load on device d (zero beyond D); the warp adds and maximises
  const uint32_t run = s.run;
  long long v = 0;
  if (tid < EB_MAX_D) {
#pragma unroll
    for (int j = 0; j < EB_MAX_MB; ++j) v += ((run >> j) & 1u) ? s.load[j][tid] : 0;
    res->joint_load[tid] = (int32_t)v;
  }
  long long num = v, peak = v;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, o);
    const long long p2 = __shfl_xor_sync(0xffffffffu, peak, o);
    peak = p2 > peak ? p2 : peak;
  }
  if (tid == 0) {
    res->run_mask = run;
    res->defer_mask = pool_mask & ~run;
    res->n_run = __popc(run);
    res->status = EB_OK;
    res->util_num = num;
    res->util_den = (long long)D * peak;
  }
}

}  // namespace
