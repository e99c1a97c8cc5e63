// Schedule(S, m) of Algorithm 1 for one thread block: the policies and the result record.
//
// MaxUtil (Section 4.2) enumerates every subset of the pool with at least m members.
// Utilisation (Eq. 3 for one step) is sum(W) / (D * max(W)); D is common to all candidates, so
// candidates are compared exactly by cross-multiplying sum and max in 64-bit integers.
// Total order: higher utilisation, then more members, then the numerically smaller mask.
// CumUtil / DiffPeak (Section 5.2) go through the pool in order, one warp with a device per lane; topping their result
// up to m members scores the remaining pool members in parallel, one lane each.
//
// What bounds small pools is latency, of large ones instruction issue: 2^16 subsets on one SM.  So there are three ways through
// the subsets of MaxUtil, none of which visits those that are too small:
//  - up to 10 members: a subset per thread; no tables, no barrier before the result is known.  The members from the sixth on are
//    the same for a whole warp, whose lanes add them up once, a device each; the other five are added member by member.
//  - more members of which few may stay out (m = ceil(0.75 n) from 12 up to n = 16: 2517 subsets): the total less the loads of
//    two pairs left out, whose sums are tabulated.
//  - otherwise the halves: the pool is split in two, and the summed load vector of each half-subset is tabulated in shared memory
//    (2 x 256 x D entries at most), so a subset costs D additions and a maximum.  The low halves are kept in the order of their
//    member counts, so that for every high half the sufficient ones come first.  Sums are 32-bit where the loads allow
//    it, and the tables' rows are 20 words apart, which 16-byte reads of neighbouring rows go through without bank conflicts.
// In a step the schedule of 4 members took 6300 cycles by halves and takes 3300 the first way, that of 12 out of 16 18000 and 11000 the
// second; 10 members is what a subset per thread of the block reaches, 4 left out what pairs and a byte per pair describe.  eb_schedule
// in a chain of its own (us, by halves / every member by itself / now): 8 members, m = 6, 16 devices 3.64 / 5.20 / 3.33, 8 devices
// 3.65 / 3.99 / 3.15; 10 members, m = 8, 16 devices 3.93 / 5.96 / 4.15 (halves take 0.5 to 1.5 more inside a step).  The pairs have
// tables of their own to lay out, which 11 members of which 1 or 2 stay out and 12 of which 1 does are too few subsets for: 3.81 / 4.06
// for 11 and 1 by halves / by pairs, 4.00 / 4.06 for 11 and 2, 3.88 / 4.00 for 12 and 1, but 4.10 / 3.99 for 12 and 2.
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
static __device__ __noinline__ Cand warp_best(Cand c) {
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
// The same for candidates whose numbers fit 32 bits and whose n is the member count of sub (or negative: none).  The quotients
// in floating point, off by less than four units in the last place, leave one candidate standing as a rule; for numbers up to
// 2048 they order like the rationals (which differ by 2^-22 of their value at least), equal ones are told apart by one more
// reduction; the rest goes through a tree of exact comparisons.  Not inlined: it is called twice.
static __device__ __noinline__ Cand warp_best_narrow(const Cand& c0) {
  int num = (int)c0.num, peak = (int)c0.peak;
  unsigned sub = c0.n < 0 ? 0u : c0.sub;   // the empty subset is never a candidate
  const unsigned key = sub ? __float_as_uint(__fdiv_rn((float)num, (float)peak)) : 0u;   // quotients of at least 1: never 0
  const unsigned top = __reduce_max_sync(0xffffffffu, key);
  unsigned left = __ballot_sync(0xffffffffu, sub != 0 && key + 8u >= top);
  const bool small = __all_sync(0xffffffffu, max(num, peak) <= 2048);
  if (__popc(left) > 1 && small) {
    const unsigned order = sub && key == top ? ((unsigned)__popc(sub) << 16 | (0xffffu ^ sub)) : 0u;
    const unsigned most = __reduce_max_sync(0xffffffffu, order);   // of one lane: subsets are distinct
    left = __ballot_sync(0xffffffffu, order == most);
  }
  if (__popc(left) > 1) {
#pragma unroll 1
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
    left = 1u;
  }
  const int at = left ? __ffs(left) - 1 : 0;   // no candidate at all: sub is 0 in every lane
  Cand c;
  c.num = __shfl_sync(0xffffffffu, num, at);
  c.peak = __shfl_sync(0xffffffffu, peak, at);
  c.sub = __shfl_sync(0xffffffffu, sub, at);
  c.n = c.sub ? __popc(c.sub) : -1;
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

// What may be left out of a pool, when that is at most kFewOut members: "pairs", the sets of at most two positions by count and
// ascending (the sets within the first np positions are the first of their count), and the sets of at most four as two pairs, the
// lower positions in the low byte, by count and ascending in the same way.
constexpr int kFewOut = 4;
constexpr int kPairs = 1 + 16 + 120;
constexpr int kFewSets = 1 + 16 + 120 + 560 + 1820;
struct FewOut {
  alignas(16) unsigned short few[(kFewSets + 7) / 8 * 8];
  alignas(16) unsigned short pair[(kPairs + 7) / 8 * 8];   // as bits
};
constexpr int single_index(int a) { return 1 + a; }
constexpr int pair_index(int a, int b) { return 17 + b * (b - 1) / 2 + a; }   // a < b
constexpr FewOut make_few_out() {
  FewOut t{};
  int at = 1;
  for (int a = 0; a < 16; ++a, ++at) {
    t.few[at] = (unsigned short)single_index(a);
    t.pair[single_index(a)] = (unsigned short)(1 << a);
  }
  for (int b = 1; b < 16; ++b)
    for (int a = 0; a < b; ++a, ++at) {
      t.few[at] = (unsigned short)pair_index(a, b);
      t.pair[pair_index(a, b)] = (unsigned short)(1 << b | 1 << a);
    }
  for (int c = 2; c < 16; ++c)
    for (int b = 1; b < c; ++b)
      for (int a = 0; a < b; ++a) t.few[at++] = (unsigned short)(pair_index(a, b) | single_index(c) << 8);
  for (int d = 3; d < 16; ++d)
    for (int c = 2; c < d; ++c)
      for (int b = 1; b < c; ++b)
        for (int a = 0; a < b; ++a) t.few[at++] = (unsigned short)(pair_index(a, b) | pair_index(c, d) << 8);
  return t;
}
static __device__ const FewOut kFew = make_few_out();

struct SchedShared {
  int4 lo[256 * kSchedRow / 4], hi[256 * kSchedRow / 4];   // summed loads of every subset of the two halves of the pool; or of pairs, and kFew
  alignas(16) int load[EB_MAX_MB][kSchedRow];              // zero beyond n_mb and D
  int nibble[4][16][EB_MAX_D];                             // summed loads of every subset of four pool positions
  unsigned char by_count[256];                             // kByCount
  int member[EB_MAX_MB];                                   // micro-batch of every pool position
  Cand best[kSchedThreads / 32];
  uint32_t run;
  bool last;                                               // this block is the last one of the grid to arrive
  long long seq_w[EB_MAX_D];
  __device__ __forceinline__ FewOut& few() { return *reinterpret_cast<FewOut*>(hi); }
  __device__ __forceinline__ const FewOut& few() const { return *reinterpret_cast<const FewOut*>(hi); }
};
static_assert(sizeof(FewOut) <= sizeof(SchedShared::hi), "the two ways through a large pool share the space");

// The best subset a thread has seen.
template <typename W>
struct BestSubset {
  W num = 0, peak = 1;
  int n = -1;
  unsigned sub = 0;
  // sum and maximum of the joint load of a subset of n2 members
  __device__ __forceinline__ void offer(W num2, W peak2, int D, int n2, unsigned sub2) {
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
  __device__ __forceinline__ Cand cand() const {
    Cand c;
    c.num = num;
    c.peak = peak;
    c.n = n;
    c.sub = sub;
    return c;
  }
};
template <typename W>
__device__ __forceinline__ W max4(W a, W b, W c, W d) {
  const W p = a > b ? a : b, q = c > d ? c : d;
  return p > q ? p : q;
}

// Best subset (pool positions as bits) of at least m members, of those this thread looks at.
// Up to 10 members.
template <typename W>
__device__ __forceinline__ Cand maxutil_small(const SchedShared& s, int D, int np, int m) {
  const int tid = threadIdx.x, lane = tid & 31, n = __popc(tid), quads = (D + 3) / 4;
  BestSubset<W> best;
  if (tid - lane < 1 << np && __popc(tid - lane) + 5 >= m) {   // else the whole warp's are too small
    W mine = 0;   // members from the sixth on are those of the whole warp: their load on device `lane` mod 16
#pragma unroll 1
    for (int k = 5; k < np; ++k)
      if ((tid >> k) & 1) mine += s.load[s.member[k]][lane & 15];
    const int4* row[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) row[k] = reinterpret_cast<const int4*>(s.load[s.member[k < np ? k : 0]]);
    W num = 0, peak = 0;
#pragma unroll 1
    for (int q = 0; q < quads; ++q) {   // entries beyond D are zero
      W w0 = 0, w1 = 0, w2 = 0, w3 = 0;
      if (np > 5) {   // a step of 4 members is 0.1 us shorter without the shuffles
        w0 = __shfl_sync(0xffffffffu, mine, 4 * q), w1 = __shfl_sync(0xffffffffu, mine, 4 * q + 1);
        w2 = __shfl_sync(0xffffffffu, mine, 4 * q + 2), w3 = __shfl_sync(0xffffffffu, mine, 4 * q + 3);
      }
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const int4 v = row[k][q];
        if ((tid >> k) & 1) {
          w0 += v.x;
          w1 += v.y;
          w2 += v.z;
          w3 += v.w;
        }
      }
      num += (w0 + w1) + (w2 + w3);
      const W p = max4(w0, w1, w2, w3);
      peak = p > peak ? p : peak;
    }
    if (tid < 1 << np && n >= m) best.offer(num, peak, D, n, tid);
  }
  return best.cand();
}
// All but at most kFewOut of up to 16 members; s.lo holds the loads of the pairs.
template <typename W>
__device__ __forceinline__ Cand maxutil_few_out(const SchedShared& s, int D, int np, int m) {
  const int tid = threadIdx.x, lane = tid & 31, quads = (D + 3) / 4, out = np - m;
  const FewOut& few = s.few();
  W mine = 0;   // total load of device `lane` mod 16
  for (int k = 0; k < np; ++k) mine += s.load[s.member[k]][lane & 15];
  const int n1 = np, n2 = n1 * (np - 1) / 2, n3 = n2 * (np - 2) / 3, n4 = n3 * (np - 3) / 4;
  const int end0 = 1, end1 = end0 + (out >= 1 ? n1 : 0), end2 = end1 + (out >= 2 ? n2 : 0), end3 = end2 + (out >= 3 ? n3 : 0),
            end4 = end3 + (out >= 4 ? n4 : 0);
  BestSubset<W> best;
#pragma unroll 1
  for (int c = tid; c - lane < end4; c += kSchedThreads) {   // whole warps go on together: the totals travel by shuffles
    const int at = c < end0 ? 0 : c < end1 ? c : c < end2 ? c - end1 + 17 : c < end3 ? c - end2 + 137 : c - end3 + 697;
    const int set = c < end4 ? few.few[at] : 0, p = set & 255, r = set >> 8;
    const int4 *x = s.lo + p * (kSchedRow / 4), *y = s.lo + r * (kSchedRow / 4);
    W num = 0, peak = 0;
    for (int q = 0; q < quads; ++q) {   // entries beyond D are zero
      const int4 a = x[q], b = y[q];
      const W w0 = __shfl_sync(0xffffffffu, mine, 4 * q) - ((W)a.x + b.x), w1 = __shfl_sync(0xffffffffu, mine, 4 * q + 1) - ((W)a.y + b.y),
              w2 = __shfl_sync(0xffffffffu, mine, 4 * q + 2) - ((W)a.z + b.z), w3 = __shfl_sync(0xffffffffu, mine, 4 * q + 3) - ((W)a.w + b.w);
      num += (w0 + w1) + (w2 + w3);
      const W p4 = max4(w0, w1, w2, w3);
      peak = p4 > peak ? p4 : peak;
    }
    const unsigned off = few.pair[p] | few.pair[r];
    if (c < end4) best.offer(num, peak, D, np - __popc(off), ((1u << np) - 1u) ^ off);
  }
  return best.cand();
}
// More than 10 members, this block's share.
template <typename W>
__device__ __forceinline__ Cand maxutil_halves(const SchedShared& s, int D, int np, int m, int block, int n_blocks) {
  const int quads = (D + 3) / 4, tid = threadIdx.x;
  static_assert(EB_MAX_D == 16 && EB_MAX_MB == 16, "the tables are indexed in nibbles");
  BestSubset<W> best;
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
      if (!(u | h)) continue;
      const int4* lo = s.lo + u * (kSchedRow / 4);
      W num = 0, peak = 0;
      for (int q = 0; q < quads; ++q) {   // entries beyond D are zero
        const int4 a = lo[q], b = hi[q];
        const W w0 = (W)a.x + b.x, w1 = (W)a.y + b.y, w2 = (W)a.z + b.z, w3 = (W)a.w + b.w;
        num += (w0 + w1) + (w2 + w3);
        const W p = max4(w0, w1, w2, w3);
        peak = p > peak ? p : peak;
      }
      best.offer(num, peak, D, n_h + __popc(u), (unsigned)(h << 8 | u));
    }
  }
  return best.cand();
}

// Whether a schedule goes the way of maxutil_few_out: 3 or 4 out of 11 members, 2 to 4 out of 12, 1 to 4 out of more.
__host__ __device__ __forceinline__ bool few_out(int np, int m, int policy) {
  return policy == EB_POLICY_MAXUTIL && np > 10 && np - m > (np < 13 ? 13 - np : 0) && np - m <= kFewOut;
}
// Whether a schedule goes through the subsets of more than 10 members.  What does not is spared their code (kLarge = false): the code
// of a kernel that runs once per step comes from far away, and what lies between costs even what never runs.
__host__ __device__ __forceinline__ bool large_pool(int np, int m, int policy) { return policy == EB_POLICY_MAXUTIL && np > 10 && np > m; }
// Which micro-batches are in the pool, and the tables that the schedule takes; before the barrier behind the writes of s.load.
__device__ __forceinline__ void schedule_prepare(SchedShared& s, uint32_t pool_mask, int m, int policy) {
  const int tid = threadIdx.x;
  if (tid < EB_MAX_MB && ((pool_mask >> tid) & 1u)) s.member[__popc(pool_mask & ((1u << tid) - 1u))] = tid;
  static_assert(sizeof(FewOut) / 16 <= kSchedThreads, "a thread per 16 bytes");
  if (few_out(__popc(pool_mask), m, policy) && tid < (int)sizeof(FewOut) / 16)
    reinterpret_cast<int4*>(&s.few())[tid] = reinterpret_cast<const int4*>(&kFew)[tid];
}
__device__ __forceinline__ bool wide_load(int v) { return v < 0 || v > kNarrowLoad; }

// Chooses the run set from s.load and returns it.  All kSchedThreads threads of the block call it after a barrier behind the writes
// of s.load and schedule_prepare; `any_wide` (uniform) unless no load is a wide_load; `block` of n_blocks; kLarge unless the schedule is
// no large_pool.  With n_blocks > 1, which is for MaxUtil over a large pool, s.best[0] is this block's candidate.  Ends with a
// barrier.
template <bool kLarge>
__device__ __forceinline__ uint32_t schedule_block(SchedShared& s, int D, uint32_t pool_mask, int m, int policy, bool any_wide, int block, int n_blocks) {
  const int tid = threadIdx.x;
  const int np = __popc(pool_mask);
  if (np <= m || policy == EB_POLICY_ALL) {
    __syncthreads();
    return pool_mask;
  }
  if (policy == EB_POLICY_MAXUTIL) {
    Cand best;
    if (!kLarge || np <= 10) {
      best = any_wide ? maxutil_small<long long>(s, D, np, m) : maxutil_small<int>(s, D, np, m);
    } else if (few_out(np, m, policy)) {
      int* pairs = reinterpret_cast<int*>(s.lo);
      for (int i = tid; i < kPairs * EB_MAX_D; i += kSchedThreads) {
        const int p = i / EB_MAX_D, d = i % EB_MAX_D;
        const unsigned bits = s.few().pair[p];
        int v = 0;
        if (bits >> np == 0) {   // the other pairs are in no set that is looked at
          if (bits) v = s.load[s.member[__ffs(bits) - 1]][d];
          if (bits & (bits - 1)) v += s.load[s.member[31 - __clz(bits)]][d];
        }
        pairs[p * kSchedRow + d] = v;
      }
      __syncthreads();
      best = any_wide ? maxutil_few_out<long long>(s, D, np, m) : maxutil_few_out<int>(s, D, np, m);
    } else {
      const int nlo = 8, nhi = np - nlo;
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
      if (tid < 64) reinterpret_cast<uint32_t*>(s.by_count)[tid] = reinterpret_cast<const uint32_t*>(kByCount.v)[tid];
      __syncthreads();
      for (int i = tid; i < (1 << nlo) * EB_MAX_D; i += kSchedThreads)
        lo[(i >> 4) * kSchedRow + (i & 15)] = s.nibble[0][(i >> 4) & 15][i & 15] + s.nibble[1][i >> 8][i & 15];
      for (int i = tid; i < (1 << nhi) * EB_MAX_D; i += kSchedThreads)
        hi[(i >> 4) * kSchedRow + (i & 15)] = s.nibble[2][(i >> 4) & 15][i & 15] + s.nibble[3][i >> 8][i & 15];
      __syncthreads();
      best = any_wide ? maxutil_halves<long long>(s, D, np, m, block, n_blocks) : maxutil_halves<int>(s, D, np, m, block, n_blocks);
    }
    // warp then block reduction under the total order (any reduction order gives the same winner), the second by one warp: all at
    // once, each for itself, they were in each other's way (800 to 1700 cycles instead of 300)
    best = any_wide ? warp_best(best) : warp_best_narrow(best);
    if ((tid & 31) == 0) s.best[tid >> 5] = best;
    __syncthreads();
    if (tid < 32) {
      best = any_wide ? warp_best(s.best[tid]) : warp_best_narrow(s.best[tid]);
      const uint32_t mask = run_mask_of(s.member, np, best);
      if (tid == 0) {
        s.run = mask;
        s.best[0] = best;
      }
    }
    __syncthreads();
    return s.run;
  }
  if (tid < 32) {
    // CumUtil / DiffPeak: ascending pool members, the first always taken; lane d holds the joint load of device d
    const int lane = tid;
    auto load_of = [&](int j) { return lane < EB_MAX_D ? (long long)s.load[j][lane] : 0LL; };
    long long w = load_of(s.member[0]);
    uint32_t chosen = 1u << s.member[0];
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
          chosen |= 1u << j;
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
        chosen |= 1u << s.member[k];
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
      if (lane < np && !((chosen >> s.member[lane]) & 1u)) {
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
      chosen |= 1u << bj;
      ++n;
    }
    if (lane == 0) s.run = chosen;
  }
  __syncthreads();
  return s.run;
}

// schedule_block by all blocks of the grid: each leaves its best candidate in global memory and the block that arrives last
// goes on with the choice among them.  False: this block is done.  The counter is ready for the next launch again.
struct SchedGrid {
  Cand* best;          // [gridDim.x]
  unsigned* arrived;
};
template <bool kLarge>
__device__ __forceinline__ bool schedule_grid(SchedShared& s, int D, uint32_t pool_mask, int m, int policy, bool any_wide, const SchedGrid& g,
                                              uint32_t* run) {
  *run = schedule_block<kLarge>(s, D, pool_mask, m, policy, any_wide, blockIdx.x, gridDim.x);
  if (!kLarge || gridDim.x == 1) return true;
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
  *run = s.run;
  return true;
}

// Blocks for a schedule: MaxUtil over the halves of a pool of more than 13 takes one per 32 high halves of its subsets.
constexpr int kMaxSchedBlocks = 1 << (EB_MAX_MB - 13);
inline int sched_blocks(uint32_t pool_mask, int m, int policy) {
  const int np = __builtin_popcount(pool_mask);
  return policy == EB_POLICY_MAXUTIL && np > m && np > 13 && !few_out(np, m, policy) ? 1 << (np - 13) : 1;
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

// The result record, by one warp.
__device__ __forceinline__ void write_schedule(const SchedShared& s, int D, uint32_t pool_mask, uint32_t run, eb_sched_result* res) {
  const int tid = threadIdx.x & 31;
  // lane d sums the chosen micro-batches' load on device d (zero beyond D); the warp adds and maximises
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

// Copies a schedule and the loads it was made from, which are written, into the record, and marks it; by one warp.  The mark is a
// release, which covers the words of the other lanes through the warp barrier, and waits until they are in host memory (1.5 us;
// with a fence of every lane before it 3 us): no other warp of a step may have to wait for this one.  Ahead of a barrier of
// tables_kernel it made a watched step of 4 x 64 tokens 32.8 us instead of 29.6; by a block of scatter_kernel of its own both are
// 29.7, and 5 x 93 tokens 91.4 -> 87.9 (unwatched 87.9).  Out of line, as calls that are not watched pay for its place in the code:
// eb_schedule of 4 members 2.98 us with it inlined, 2.83 without.
static __device__ __noinline__ void leave_record(const ScheduleWatch& watch, const eb_sched_result* res, const int32_t* load, int n_load) {
  const int lane = threadIdx.x & 31;
  static_assert(sizeof(eb_sched_result) % 4 == 0 && sizeof(eb_sched_result) / 4 <= 32, "a word per lane");
  if (lane < (int)sizeof(eb_sched_result) / 4) reinterpret_cast<int32_t*>(&watch.rec->res)[lane] = reinterpret_cast<const int32_t*>(res)[lane];
  for (int i = lane; i < n_load; i += 32) watch.rec->load[i] = load[i];
  __syncwarp();
  if (lane == 0) asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(&watch.rec->ticket), "r"(watch.ticket) : "memory");
}

}  // namespace
