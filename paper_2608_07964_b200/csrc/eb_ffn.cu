// eb_expert_ffn_grouped: expert_i of Eq. 1 (bias-free SwiGLU MLP) for every (layer, expert) group
// of a step in one grouped pass on the 5th-generation tensor cores.
//
// One persistent launch over a device-built tile list (ragged groups, no padding rows in memory), gate/up
// tiles first, down tiles after them in the same order of groups:
//   gate/up : act[r, i] = silu(sum_h xp[r,h] Wg[i,h]) * (sum_h xp[r,h] Wu[i,h])      (bf16 out)
//   down    : yp[r, h]  = sum_i act[r,i] Wd[h,i]                                      (bf16 out)
//
// ffn_kernel runs on CTA pairs (2-CTA clusters, one CTA per SM).  The WEIGHTS are the M operand of
// tcgen05.mma cta_group::2 (M = 256 weight rows, 128 per CTA) and the TOKEN rows of the tile are the N
// operand: N = the tile's rows rounded up to 16, at most 256.  Tensor-core work, shared-memory fill and
// TMEM columns of a tile therefore follow the rows it really holds - a group of 45 rows costs a 48-column
// tile, not a 128- or 256-row one - and a group is cut into ceil(rows / 256) tiles of nearly equal size.
// Every k-step issues two MMAs that share the token operand:
//   gate/up: W0 = 256 rows of W_gate, W1 = the same 256 rows of W_up.  The TMEM lane that holds gate
//            output i of a token holds up output i of that token, so SiLU * up fuses in registers
//            (256 outputs per tile);
//   down   : W0, W1 = two consecutive 256-row blocks of W_down (512 outputs per tile).
// Per CTA: warp 0 = TMA producer (its own 128 rows of W0 and W1 and its half of the token rows), warp 1 =
// MMA issuer (leader CTA only) and TMEM owner, warps 2..9 = epilogue, warp 10 = publisher of finished rows.  A stage is 48 KB per CTA (W0 | W1 |
// up to 128 token rows of one 64-wide k-block, bf16, 128-byte swizzled K-major) for up to 1024 tensor-core
// cycles; four stages.  TMA completions of both CTAs count on the leader's barrier; the tcgen05.commit
// that frees a stage is delivered to both CTAs; no load is multicast.
//
// Epilogue against the next tile's MMAs.  The two accumulators of a tile of more than 128 columns fill TMEM
// (2 x 256 fp32 columns).  What bounds such a tile is then how soon the accumulators come back: the eight
// epilogue warps (two per lane quadrant, alternating 16-column chunks) read the whole first accumulator into
// registers and hand it back, then the second one, and only then transpose and store; the MMA warp starts the
// next tile with the first accumulator alone, over the k-blocks that the ring holds, and follows up with the
// second.  Storing chunk by chunk before handing anything back kept the tensor pipe idle for 6100 cycles per
// tile (of 36000 in gate/up, 29000 in down at H 2048, I 1408), this order for 1900: the expert pass of 49152
// rows over 66 matrices went from 725 to 689 us.  Tiles of at most 128 columns take one half of TMEM in turn,
// so their epilogue runs beside the next tile's MMAs (16-434 rows a group over 788 matrices: 2245 -> 2236 us).
// The accumulator holds outputs in lanes and tokens in columns: an epilogue warp transposes each 16-token
// chunk through 1 KB of shared memory and stores 16-byte vectors.
//
// Tiles: a device-built list (eb_tiles.cuh).  Tiles of one group are weight-tile-major and
// token-tile-minor, so pairs working side by side share the weight tile in L2 and every weight byte leaves
// HBM once per group.  The D replicas of a shared expert (one group per virtual device, all reading the
// same matrix) are merged when all are small: their rows are packed into common tiles in slots of 16
// rows, so the matrix is streamed once per step instead of D times.  Groups are listed widest tiles
// first; every pair takes the next tile of the list when it is nearly through with the one before (a dealer
// thread per pair claims it and leaves it in both CTAs' mailboxes).  A down tile starts when the gate/up tiles
// of its rows are counted complete; those were dealt earlier, to pairs that are running, so every wait ends.
// With a launch per phase and tiles dealt out beforehand, pairs that were through waited for the last one twice
// per step (20 us of 240 in gate/up, 13 of 130 in down at 133 matrices of 3 x 2048 x 1408) and the down launch
// began with an empty ring: the expert pass took 372 us there, 116 at 126 matrices of 3 x 1000 x 712 and 109 at
// 32 of the former, this way 361, 105 and 102.
//
// Every wait on an mbarrier is bounded: on expiry the kernel records EB_ERR_TIMEOUT in the
// context status word, lets copies in flight land, frees its TMEM and returns.
#include <cstddef>
#include <type_traits>

#include "eb_tiles.cuh"

namespace {

constexpr int BK = 64;                                         // bf16 elements of one k-block (128 bytes)
constexpr int kStages = 4;
constexpr int kWBytes = 128 * BK * 2;                          // 128 weight rows of one k-block
constexpr int kTBytes = 128 * BK * 2;                          // up to 128 token rows of one k-block
constexpr int kStageBytes = 2 * kWBytes + kTBytes;             // W0 | W1 | token rows
constexpr int kRingBytes = kStages * kStageBytes;
constexpr int kEpiWarps = 8;                                   // two per TMEM lane quadrant
constexpr int kThreads = 96 + 32 * kEpiWarps;
constexpr int kChunkStep = 16 * (kEpiWarps / 4);               // columns between two chunks of an epilogue warp
constexpr size_t kSmemBytes = (size_t)kRingBytes + 1024 /*alignment slack*/ + 512 /*barriers*/ + kEpiWarps * 1024 /*transposes*/;
static_assert(kSmemBytes <= 232448, "shared memory of one CTA");
constexpr int kTmemCols = 512;
constexpr int kTmemHalf = 256;                                 // a narrow tile's two accumulators share one half of TMEM
constexpr int kNarrowCols = kTmemHalf / 2;                     // ... which takes tiles of up to 128 columns
constexpr int kItems = 2;                                      // mailbox slots of a CTA (tiles dealt ahead)
constexpr int kParts = 4;                                      // tiles whose epilogues may be under way at once in a CTA: a tile is dealt
                                                               // only when every reader has taken the one kItems before it, so at most kItems + 1
static_assert(kParts > kItems, "a barrier of the publisher is free again before it comes round");
constexpr int kAskAhead = 16;                                  // k-blocks before the end of a tile at which its successor is asked for
constexpr long long kSpinLimitCycles = 4000000000LL;

// ---- PTX wrappers ----------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// whether the phase is over, without waiting
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded waits: false if the limit expired or another thread of the CTA already gave up.
template <typename Try>
__device__ __forceinline__ bool bounded_wait(Try try_once, volatile int* s_abort, int* status, long long limit = kSpinLimitCycles) {
  if (try_once()) return true;
  const long long t0 = clock64();
  for (uint32_t spin = 1;; ++spin) {
    if (try_once()) return true;
    if ((spin & 63u) == 0u) {
      if (*s_abort) return false;
      if (clock64() - t0 > limit) {
        *s_abort = 1;
        atomicExch(status, (int)EB_ERR_TIMEOUT);
        return false;
      }
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* s_abort, int* status,
                                          long long limit = kSpinLimitCycles) {
  return bounded_wait([&] { return mbar_try(bar, parity); }, s_abort, status, limit);
}
// the same for a barrier that the peer CTA's ordinary stores arrive with
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* s_abort, int* status) {
  return bounded_wait([&] { return mbar_try_cluster(bar, parity); }, s_abort, status);
}

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of the same offset in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Says "done with it" to a barrier of the pair: nothing this thread wrote is handed over.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// Hands what the warp wrote to a thread of the same CTA.
__device__ __forceinline__ void mbar_arrive_release(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// The same as mbar_arrive_cluster with what this thread wrote before it.  Only the tile dealer uses it: a release at cluster scope waits for
// the thread's earlier accesses, and in the producer, MMA and epilogue warps that cost 1 to 2 us per tile.
__device__ __forceinline__ void mbar_arrive_release_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t cluster_addr, const int4& v) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ int4 ld_shared(uint32_t addr) {
  int4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Counts one up; what the thread has seen written goes before (release: a fence and a relaxed addition).  Between the two, what it has
// seen is also put before later accesses of TMA units.  A step of 4 x 64 tokens, where every down tile waits for this, 33.5 -> 33.2 us
// against a __threadfence and a red.release.
__device__ __forceinline__ void red_publish(int* p) {
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  asm volatile("fence.proxy.async;" ::: "memory");
  asm volatile("red.relaxed.gpu.global.add.s32 [%0], 1;" ::"l"(p) : "memory");
}
// orders ordinary memory accesses with those of the TMA unit
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async;" ::: "memory"); }
// TMA loads whose completion is counted on a barrier that may live in the peer CTA (the data goes to the
// issuing CTA only)
__device__ __forceinline__ void tma_pair_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_pair_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
// D[tmem of both CTAs] (+)= A * B^T with M = 256 (128 rows of A per CTA), N from the descriptor (half of B per CTA), K = 16
__device__ __forceinline__ void umma_pair_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5, %5, %5, %5, %5}, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(0u)
      : "memory");
}
// arrives on the barrier at this offset in both CTAs of the pair once the MMAs issued so far are done
__device__ __forceinline__ void umma_pair_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"((uint16_t)3)
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }



__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory operand descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// Instruction descriptor: fp32 accumulate, bf16 A and B, both K-major; M weight rows and N token columns.
__device__ __forceinline__ uint32_t instr_desc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// silu(g) * u with one special-function instruction: silu(g) = g / (1 + exp(-g)) = h + h tanh(h), h = g / 2.
// tanh.approx.f32 is good to about 2^-11 relative, well inside the bf16 rounding of the result.
__device__ __forceinline__ float silu_mul(uint32_t g_bits, uint32_t u_bits) {
  const float h = 0.5f * __uint_as_float(g_bits), u = __uint_as_float(u_bits);
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(h));
  return fmaf(h, t, h) * u;
}

// A gate/up tile with at most 128 outputs left (the last of I = 1408: eleven times 128) is multiplied with M = 128, 64
// weight rows per CTA: the tensor cores then spend half the time on it instead of working on 128 rows of zeros.  The
// accumulator of such an MMA holds the CTA's 64 outputs twice over in its lanes, each time for half of the tokens.
// At 49152 rows over 66 matrices of 3 x 2048 x 1408 the step went from 926 to 908 us, the expert pass alone from 698 to
// 682; where weights are streamed nothing changes.
__device__ __forceinline__ bool slim_tile(int n_out, int out) { return n_out - out * kFeat1 <= kFeat1 / 2; }

// Which part of TMEM a tile's two accumulators take.  TMEM is two halves of 256 columns, each with a full and an
// empty barrier.  A tile of more than 128 columns takes both (one accumulator in each); a narrower one takes the
// half that is next in turn, so that its epilogue runs while the next tile's MMAs fill the other half.  The MMA
// warp and the epilogue warps walk the same tiles and so reach the same placement and the same barrier phases.
struct TmemTurn {
  uint32_t used = 0;      // bits 0, 1: halves of the current tile; bit 2: the half whose turn is next
  uint32_t phases = 3;    // bit h: phase parity of the current use of half h (the first use has parity 0)
  __device__ __forceinline__ void take(int cols) {
    const uint32_t next = used >> 2;
    used = cols > kNarrowCols ? (3u | (next << 2)) : ((1u << next) | ((next ^ 1u) << 2));
    phases ^= used & 3u;
  }
  __device__ __forceinline__ bool wide() const { return (used & 3u) == 3u; }
  __device__ __forceinline__ int half() const { return (int)((used >> 1) & 1u); }   // of a narrow tile
  __device__ __forceinline__ uint32_t parity(int h) const { return (phases >> h) & 1u; }
  __device__ __forceinline__ uint32_t col0() const { return (used & 3u) == 2u ? kTmemHalf : 0; }
  __device__ __forceinline__ uint32_t step() const { return (used & 3u) == 3u ? kTmemHalf : kNarrowCols; }
};

// An epilogue warp whose TMEM reads are complete (wait::ld) hands its part of an accumulator back to the MMA warp.
__device__ __forceinline__ void release_tmem(uint32_t bar, int lane) {
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive_cluster(map_to_cta(bar, 0));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ bf16 low_half(uint32_t v) { return __ushort_as_bfloat16((unsigned short)(v & 0xffffu)); }
__device__ __forceinline__ bf16 high_half(uint32_t v) { return __ushort_as_bfloat16((unsigned short)(v >> 16)); }

// Chunks at columns 0, kChunkStep, .. of an accumulator, rounded to bf16, two tokens per word.
template <int N>
__device__ __forceinline__ void drain_packed(uint32_t acc, uint32_t (&out)[N][8]) {
  constexpr int P = N < 2 ? 1 : 2;   // loads in flight
#pragma unroll
  for (int i = 0; i < N; i += P) {
    uint32_t a[P][16];
#pragma unroll
    for (int k = 0; k < P; ++k) tmem_ld16(acc + kChunkStep * (i + k), a[k]);
    tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < P; ++k)
#pragma unroll
      for (int j = 0; j < 8; ++j) out[i + k][j] = pack_bf16(__uint_as_float(a[k][2 * j]), __uint_as_float(a[k][2 * j + 1]));
  }
}

// ---- the grouped GEMM kernel -----------------------------------------------------------------
// Token-row boxes of 128 / 64 / 32 / 16 / 8 rows over one activation tensor.
struct TokenMaps {
  CUtensorMap box[5];
};
struct FfnParams {
  TokenMaps xp, act;                 // inputs of the two phases
  CUtensorMap gate, up, down;        // weight boxes of 128 rows
  CUtensorMap gate64, up64;          // of 64 rows; with the above kMaps tensor maps in a row
  const Tile* work;                  // the list: gate/up tiles, then down tiles
  const int2* slots;
  const int32_t* work_count;         // [0], [1]: tiles of the two phases
  int32_t* next;                     // tiles dealt out (second entry: of a launch of part 2)
  int32_t* ready;                    // per token tile: arrivals, one per CTA for every finished gate/up tile
  bf16 *act_out, *yp;
  int H, I;
  int part;                          // 0: the whole list; 1, 2: the tiles of that phase only
  int* status;
};

constexpr int kMaps = 15;
static_assert(offsetof(FfnParams, up64) == (kMaps - 1) * sizeof(CUtensorMap), "the maps are prefetched as an array");

// Chunks of 16 token columns of a finished tile: registers -> transposed through shared memory -> rows.  NC chunks
// of this warp are read, of which those below the tile's columns hold rows (every chunk read lies in the accumulator).
// The tile's token columns token0 .. token0 + tmem_cols - 1 lie in this warp's accumulator columns 0 ..; the rows of a
// chunk at token column c are row0 .. row0 + n_here - 1 (a merged tile: one slot).
// Global stores are 16-byte vectors: lane -> (token lane / 4 (+8), outputs 8 (lane % 4) .. +7).
template <int PHASE, int NC>
__device__ __forceinline__ void epilogue_tile(const Tile& it, const TmemTurn& turn, uint32_t taddr, int chunk0, int lane, int fbase,
                                              int token0, int tmem_cols, bf16* tile, const int2* __restrict__ slots, bf16* __restrict__ out, int n_out,
                                              uint32_t tempty0, uint32_t tempty1) {
  const bool merged = it.rows < 0;
  const int n_cols = merged ? -it.rows * kSlotRows : it.rows;   // columns that may hold rows to store
  const uint32_t acc0 = taddr + turn.col0() + chunk0, acc1 = acc0 + turn.step();
  // chunk i of one accumulator, two tokens per word, to its rows; its outputs start at column f
  auto store_chunk = [&](const uint32_t* v, int i, int f) {
    const int left = tmem_cols - (chunk0 + kChunkStep * i), c = token0 + chunk0 + kChunkStep * i;
    if (left > 0 && c < n_cols) {
      int row0 = it.row + c, n_here = min(min(16, left), it.rows - c);
      if (merged) {
        const int2 sl = __ldg(slots + it.row + (c >> 4));
        row0 = sl.x;
        n_here = sl.y;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        tile[2 * j * 32 + lane] = low_half(v[j]);
        tile[(2 * j + 1) * 32 + lane] = high_half(v[j]);
      }
      __syncwarp();
      const int fcol = f + (lane & 3) * 8;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int tok = (lane >> 2) + 8 * h;
        if (tok < n_here && fcol < n_out)
          *reinterpret_cast<uint4*>(out + (size_t)(row0 + tok) * n_out + fcol) =
              *reinterpret_cast<const uint4*>(tile + tok * 32 + (lane & 3) * 8);
      }
      __syncwarp();
    }
  };
  // The accumulators move to registers, rounded (down) or combined (gate/up), and are handed back as soon as they are
  // read; the stores come after.
  const uint32_t tempty_last = turn.wide() || turn.half() ? tempty1 : tempty0;
  if constexpr (PHASE == 1) {
    uint32_t r[NC][16];   // the gate accumulator; then outputs in [0..7]
#pragma unroll
    for (int i = 0; i < NC; ++i) tmem_ld16(acc0 + kChunkStep * i, r[i]);
    tmem_ld_wait();
    if (turn.wide()) release_tmem(tempty0, lane);
#pragma unroll
    for (int i = 0; i < 2 * NC; ++i) {   // eight columns at a time: no register is left for more
      uint32_t b[8];
      uint32_t* const g = r[i / 2] + (i % 2) * 8;
      tmem_ld8(acc1 + kChunkStep * (i / 2) + (i % 2) * 8, b);
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < 4; ++j)
        r[i / 2][(i % 2) * 4 + j] = pack_bf16(silu_mul(g[2 * j], b[2 * j]), silu_mul(g[2 * j + 1], b[2 * j + 1]));
    }
    release_tmem(tempty_last, lane);
#pragma unroll
    for (int i = 0; i < NC; ++i) store_chunk(r[i], i, fbase);
  } else {
    uint32_t r0[NC][8], r1[NC][8];
    drain_packed(acc0, r0);
    if (turn.wide()) release_tmem(tempty0, lane);
    // half of it is stored while the next tile's first MMAs run, which makes room for the second accumulator
#pragma unroll
    for (int i = 0; i < NC / 2; ++i) store_chunk(r0[i], i, fbase);
    drain_packed(acc1, r1);
    release_tmem(tempty_last, lane);
#pragma unroll
    for (int i = NC / 2; i < NC; ++i) store_chunk(r0[i], i, fbase);
#pragma unroll
    for (int i = 0; i < NC; ++i) store_chunk(r1[i], i, fbase + 256);
  }
}

__global__ void __launch_bounds__(kThreads, 1)
ffn_kernel(const __grid_constant__ FfnParams p) {
  EB_GRID_DEP_SYNC();
  constexpr int NS = kStages;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);
  const uint32_t bar0 = base + (uint32_t)kRingBytes;
  auto w0_addr = [&](int s) { return base + s * kStageBytes; };
  auto w1_addr = [&](int s) { return base + s * kStageBytes + kWBytes; };
  auto t_addr = [&](int s) { return base + s * kStageBytes + 2 * kWBytes; };
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (NS + s); };
  auto tfull_bar = [&](int h) { return bar0 + 8u * (2 * NS + h); };
  auto tempty_bar = [&](int h) { return bar0 + 8u * (2 * NS + 2 + h); };
  auto item_full = [&](int i) { return bar0 + 8u * (2 * NS + 4 + i); };
  auto item_empty = [&](int i) { return bar0 + 8u * (2 * NS + 4 + kItems + i); };
  const uint32_t want_bar = bar0 + 8u * (2 * NS + 4 + 2 * kItems);
  auto part_bar = [&](int i) { return bar0 + 8u * (2 * NS + 4 + 2 * kItems + 1 + i); };
  constexpr int kBarBytes = 8 * (2 * NS + 4 + 2 * kItems + 1 + kParts), kMailbox = 512 - kItems * (int)sizeof(Tile);
  static_assert(kBarBytes + 8 <= kMailbox, "512 bytes of barriers and mailbox");
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(smem + kRingBytes + kBarBytes);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + kRingBytes + kBarBytes + 4);
  const uint32_t items = bar0 + kMailbox;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();   // CTA 0 of a pair is the leader
  int* const status = p.status;
  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(full_bar(s), 1);    // the leader's arrive + all bytes of the stage of both CTAs
      mbar_init(empty_bar(s), 1);   // one tcgen05.commit (delivered to both CTAs)
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(tfull_bar(h), 1);                // one tcgen05.commit
      mbar_init(tempty_bar(h), 2 * kEpiWarps);   // one arrival per epilogue warp of both CTAs (leader's barrier)
    }
    for (int i = 0; i < kItems; ++i) {
      mbar_init(item_full(i), 1);                        // the dealer's arrive
      mbar_init(item_empty(i), 5 + 2 * kEpiWarps);       // every reader of both CTAs (CTA 1's barrier)
    }
    for (int i = 0; i < kParts; ++i) mbar_init(part_bar(i), kEpiWarps);   // one arrival per epilogue warp of the CTA
    mbar_init(want_bar, 1);                              // the leader's producer (CTA 1's barrier)
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2 && lane < kMaps) prefetch_tmap(&p.xp.box[0] + lane);
  // The pair's first tile, claimed like all others: were it fixed beforehand, a pair that cannot run yet (another
  // kernel of this kind holds its SMs) would keep it, and both kernels could wait for such tiles.  One thread of CTA 1
  // claims it, so that the trip to memory passes beside the set-up.
  int4 first_a = make_int4(0, 0, -1, 0), first_b = make_int4(0, 0, 0, 0);
  const bool claims_first = rank == 1 && threadIdx.x == 96;
  if (claims_first) {
    const int cnt1 = p.work_count[0], cnt2 = p.work_count[1];
    const int idx = (p.part == 2 ? cnt1 : 0) + atomicAdd(p.next + (p.part == 2 ? 1 : 0), 1);
    if (idx < (p.part == 1 ? cnt1 : cnt1 + cnt2)) {
      const int4* e = reinterpret_cast<const int4*>(p.work + idx);
      first_a = __ldg(e);
      first_b = __ldg(e + 1);
    }
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32((const void*)s_tmem), kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // the peer's barriers are initialised before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;
  const int num_kb1 = (p.H + BK - 1) / BK, num_kb2 = (p.I + BK - 1) / BK;

  // leaves a tile in slot i of both CTAs' mailboxes
  auto deal = [&](int i, const int4& a, const int4& b) {
    for (uint32_t r = 0; r < 2; ++r) {
      const uint32_t dst = map_to_cta(items + i * (uint32_t)sizeof(Tile), r);
      st_cluster(dst, a);
      st_cluster(dst + 16, b);
      mbar_arrive_release_cluster(map_to_cta(item_full(i), r));
    }
  };
  if (claims_first) deal(0, first_a, first_b);
  // Tile number `seq` of this pair, from the mailbox (false: gave up); the reader then frees the slot.
  auto take_item = [&](int seq, Tile* it) {
    const int i = seq % kItems;
    if (!mbar_wait_cluster(item_full(i), (uint32_t)(seq / kItems) & 1u, s_abort, status)) return false;
    const int4 a = ld_shared(items + i * (uint32_t)sizeof(Tile)), b = ld_shared(items + i * (uint32_t)sizeof(Tile) + 16);
    *it = Tile{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    return true;
  };
  auto free_item = [&](int seq) { mbar_arrive_cluster(map_to_cta(item_empty(seq % kItems), 1)); };

  if (warp == 0) {
    // ---------------- TMA producer (each CTA loads its own halves) ----------------
    if (lane == 0) {
      // A weight tile that one tile alone reads goes through L2 as the first to leave it: left to the usual policy, the
      // stream of weights pushes out the rows, the tables and the code of the small kernels, which then start from
      // HBM in every step (133 matrices of 3 x 2048 x 1408: 388 -> 363 us a step, 359 -> 343 of it in this kernel).  Tiles
      // that share weights keep them: evicted early, they cost 1-2 % at several hundred rows per group.
      uint64_t stream_policy, keep_policy;
      asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(stream_policy));
      asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(keep_policy));
      int stage = 0;
      uint32_t phase = 0;
      for (int seq = 0;; ++seq) {
        Tile it;
        if (!take_item(seq, &it)) goto done;
        if (it.w < 0) break;
        free_item(seq);
        const uint64_t w_policy = it.once ? stream_policy : keep_policy;
        const bool merged = it.rows < 0;
        const int half = entry_cols(it.rows) >> 1;   // token rows this CTA loads: a multiple of 8 (of 16 in a merged tile)
        const int tok0 = it.row + (int)rank * half;
        // merged tile: this CTA's slots are slots[row + rank * half / 16 ..); a slot beyond the tile's count
        // repeats the first one (its columns are never stored), so the byte count of a stage stays uniform
        int slot_row[kMergeSlots / 2];
#pragma unroll
        for (int i = 0; i < kMergeSlots / 2; ++i) {
          const int sl = (int)rank * (half / kSlotRows) + i;
          slot_row[i] = (merged && i < half / kSlotRows) ? __ldg(p.slots + it.row + (sl < -it.rows ? sl : 0)).x : 0;
        }
        const bool down = it.phase == 2;
        const CUtensorMap* tmW0 = down ? &p.down : &p.gate;
        const CUtensorMap* tmW1 = down ? &p.down : &p.up;
        const TokenMaps* tmT = down ? &p.act : &p.xp;
        const int num_kb = down ? num_kb2 : num_kb1;
        const bool slim = !down && slim_tile(p.I, it.out);   // 64 weight rows per CTA and operand
        if (slim) {
          tmW0 = &p.gate64;
          tmW1 = &p.up64;
        }
        const int wrow0 = it.out * (down ? kFeat2 : kFeat1) + (int)rank * (slim ? 64 : 128);
        const int wrow1 = down ? wrow0 + 256 : wrow0;
        const uint32_t tx = 2u * ((slim ? 1u : 2u) * kWBytes + (uint32_t)half * (BK * 2));
        // both CTAs' copies are counted on the leader's barrier; the leader announces the total
        auto load_weights = [&](int st, int kb) {
          const uint32_t fb = map_to_cta(full_bar(st), 0);
          if (rank == 0) mbar_expect_tx(full_bar(st), tx);
          tma_pair_load_3d(w0_addr(st), tmW0, kb * BK, wrow0, it.w, fb, w_policy);
          tma_pair_load_3d(w1_addr(st), tmW1, kb * BK, wrow1, it.w, fb, w_policy);
        };
        auto load_tokens = [&](int st, int kb) {
          const uint32_t fb = map_to_cta(full_bar(st), 0), ta = t_addr(st);
          if (merged) {
#pragma unroll
            for (int i = 0; i < kMergeSlots / 2; ++i)
              if (i < half / kSlotRows) tma_pair_load_2d(ta + i * (kSlotRows * BK * 2), &tmT->box[3], kb * BK, slot_row[i], fb);
          } else if (half == 128) {
            tma_pair_load_2d(ta, &tmT->box[0], kb * BK, tok0, fb);
          } else {
            int r2 = 0;   // rows placed so far; every box starts on a multiple of 8 rows (1 KB), which keeps the swizzle phase
            if (half & 64) {
              tma_pair_load_2d(ta, &tmT->box[1], kb * BK, tok0, fb);
              r2 = 64;
            }
            if (half & 32) {
              tma_pair_load_2d(ta + r2 * (BK * 2), &tmT->box[2], kb * BK, tok0 + r2, fb);
              r2 += 32;
            }
            if (half & 16) {
              tma_pair_load_2d(ta + r2 * (BK * 2), &tmT->box[3], kb * BK, tok0 + r2, fb);
              r2 += 16;
            }
            if (half & 8) tma_pair_load_2d(ta + r2 * (BK * 2), &tmT->box[4], kb * BK, tok0 + r2, fb);
          }
        };
        const int ask = num_kb > kAskAhead ? num_kb - kAskAhead : 0;
        int kb = 0;
        if (down) {
          const int* flag = p.ready + it.done;
          if (it.need > 0 && ld_acquire(flag) < it.need) {
            // the rows are still being made: the weights of the stages at hand go ahead of them
            const int lead = num_kb < NS ? num_kb : NS;
            int st = stage;
            uint32_t ph = phase;
            for (int i = 0; i < lead; ++i) {
              if (!mbar_wait(empty_bar(st), ph ^ 1u, s_abort, status)) goto done;
              load_weights(st, i);
              if (++st == NS) {
                st = 0;
                ph ^= 1u;
              }
            }
            if (!bounded_wait([&] { return ld_acquire(flag) >= it.need; }, s_abort, status)) goto done;
            fence_proxy_async();
            if (rank == 0 && ask < lead) mbar_arrive_cluster(map_to_cta(want_bar, 1));
            for (; kb < lead; ++kb) {
              load_tokens(stage, kb);
              if (++stage == NS) {
                stage = 0;
                phase ^= 1u;
              }
            }
          } else {
            fence_proxy_async();
          }
        }
        for (; kb < num_kb; ++kb) {
          if (rank == 0 && kb == ask) mbar_arrive_cluster(map_to_cta(want_bar, 1));
          if (!mbar_wait(empty_bar(stage), phase ^ 1u, s_abort, status)) goto done;
          load_weights(stage, kb);
          load_tokens(stage, kb);
          if (++stage == NS) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      // ---------------- MMA issuer (leader CTA only) ----------------
      int stage = 0;
      uint32_t phase = 0;
      TmemTurn turn;
      for (int seq = 0;; ++seq) {
        Tile it;
        if (!take_item(seq, &it)) goto done;
        if (it.w < 0) break;
        free_item(seq);
        const int num_kb = it.phase == 2 ? num_kb2 : num_kb1;
        const int cols = entry_cols(it.rows);
        const uint32_t idesc = instr_desc(it.phase == 1 && slim_tile(p.I, it.out) ? 128 : 256, cols);
        turn.take(cols);
        const uint32_t acc0 = tmem_base + turn.col0(), acc1 = acc0 + turn.step();
        int kb = 0;
        if (turn.wide() && !mbar_test(tempty_bar(1), turn.parity(1) ^ 1u)) {
          // the epilogue hands the first accumulator back well before the second: the k-blocks that fit the ring
          // are multiplied into the first one, then into the second, then both go on together.  Not when both are free
          // already: the stages come back later this way (one tile per pair and phase, 256 rows, 16 and 12 k-blocks: 44.5 us
          // for the pass instead of 42.6)
          const int lead = num_kb < NS ? num_kb : NS;
          if (!mbar_wait(tempty_bar(0), turn.parity(0) ^ 1u, s_abort, status)) goto done;
          tc_fence_after();
          int st = stage;
          uint32_t ph = phase;
          for (int i = 0; i < lead; ++i) {
            if (!mbar_wait(full_bar(st), ph, s_abort, status)) goto done;
            tc_fence_after();
            const uint64_t d0 = smem_desc(w0_addr(st)), dt = smem_desc(t_addr(st));
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) umma_pair_bf16(acc0, d0 + 2 * k, dt + 2 * k, idesc, (i | k) != 0 ? 1u : 0u);
            if (++st == NS) {
              st = 0;
              ph ^= 1u;
            }
          }
          if (!mbar_wait(tempty_bar(1), turn.parity(1) ^ 1u, s_abort, status)) goto done;
          tc_fence_after();
          for (; kb < lead; ++kb) {
            const uint64_t d1 = smem_desc(w1_addr(stage)), dt = smem_desc(t_addr(stage));
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) umma_pair_bf16(acc1, d1 + 2 * k, dt + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
            umma_pair_commit(empty_bar(stage));
            if (++stage == NS) {
              stage = 0;
              phase ^= 1u;
            }
          }
        } else {
          const int h = turn.wide() ? 0 : turn.half();
          if (!mbar_wait(tempty_bar(h), turn.parity(h) ^ 1u, s_abort, status)) goto done;
          tc_fence_after();
        }
        for (; kb < num_kb; ++kb) {
          if (!mbar_wait(full_bar(stage), phase, s_abort, status)) goto done;
          tc_fence_after();
          const uint64_t d0 = smem_desc(w0_addr(stage)), d1 = smem_desc(w1_addr(stage)), dt = smem_desc(t_addr(stage));
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            umma_pair_bf16(acc0, d0 + 2 * k, dt + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
            umma_pair_bf16(acc1, d1 + 2 * k, dt + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
          }
          umma_pair_commit(empty_bar(stage));   // the stage is reusable in both CTAs once these MMAs have read it
          if (++stage == NS) {
            stage = 0;
            phase ^= 1u;
          }
        }
        // both accumulators complete
        if (turn.wide()) {
          umma_pair_commit(tfull_bar(0));
          umma_pair_commit(tfull_bar(1));
        } else {
          umma_pair_commit(tfull_bar(turn.half()));
        }
      }
    } else if (lane == 0) {
      // ---------------- tile dealer (CTA 1's otherwise idle MMA warp) ----------------
      // Every further tile of a pair is the next one not yet dealt, claimed well before the leader's producer is
      // through with the tile before it.
      const int part_first = p.part == 2 ? p.work_count[0] : 0;
      const int part_end = p.part == 1 ? p.work_count[0] : p.work_count[0] + p.work_count[1];
      Tile it;
      if (!take_item(0, &it)) goto done;
      for (int seq = 1; it.w >= 0; ++seq) {
        const int i = seq % kItems;
        if (!mbar_wait_cluster(want_bar, (uint32_t)(seq - 1) & 1u, s_abort, status)) goto done;
        if (seq >= kItems && !mbar_wait_cluster(item_empty(i), (uint32_t)(seq / kItems - 1) & 1u, s_abort, status)) goto done;
        const int idx = part_first + atomicAdd(p.next + (p.part == 2 ? 1 : 0), 1);
        int4 a = make_int4(0, 0, -1, 0), b = make_int4(0, 0, 0, 0);
        if (idx < part_end) {
          const int4* e = reinterpret_cast<const int4*>(p.work + idx);
          a = __ldg(e);
          b = __ldg(e + 1);
          // a down tile whose rows are complete already, the usual case, spares the producers the question
          if (b.x == 2 && ld_acquire(p.ready + b.y) >= b.z) b.z = 0;
        }
        deal(i, a, b);
        if (idx >= part_end) break;
      }
    }
  } else if (warp == 2 + kEpiWarps) {
    if (lane == 0) {
      // ---------------- publisher: counts the CTA's share of a finished gate/up tile on its token tile ----------------
      // The down tiles of these rows wait for all shares.  The epilogue warps' stores are ordered before the TMA reads of
      // whoever sees the count.  A thread of its own, since the fence waits for those stores: in the CTA's last epilogue warp it
      // held up the next tile's epilogue, 98 instead of 89 us at 49152 rows over 132 matrices of 3 x 256 x 512.
      uint32_t uses = 0;   // bit i: phase parity of the next use of part_bar(i)
      for (int seq = 0;; ++seq) {
        Tile it;
        if (!take_item(seq, &it)) goto done;
        if (it.w < 0) break;
        free_item(seq);
        if (it.phase != 1) continue;
        const int i = seq % kParts;
        if (!mbar_wait(part_bar(i), (uses >> i) & 1u, s_abort, status)) goto done;
        uses ^= 1u << i;
        red_publish(p.ready + it.done);
      }
    }
  } else {
    // ---------------- epilogue warps ----------------
    const int q = warp & 3;                      // TMEM lane quadrant this warp may read
    const int chunk0 = ((warp - 2) >> 2) * 16;   // the warps of a quadrant take 16-column chunks in turn
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16);
    bf16* tile = reinterpret_cast<bf16*>(smem + kRingBytes + 512) + (warp - 2) * 512;   // 1 KB per epilogue warp
    TmemTurn turn;
    for (int seq = 0;; ++seq) {
      // one lane waits, the outcome is made warp-uniform before any .aligned instruction
      Tile it = {};
      int ok = 1;
      if (lane == 0) ok = take_item(seq, &it) ? 1 : 0;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) goto done;
      it.row = __shfl_sync(0xffffffffu, it.row, 0);
      it.rows = __shfl_sync(0xffffffffu, it.rows, 0);
      it.w = __shfl_sync(0xffffffffu, it.w, 0);
      it.out = __shfl_sync(0xffffffffu, it.out, 0);
      it.phase = __shfl_sync(0xffffffffu, it.phase, 0);
      if (it.w < 0) break;
      turn.take(entry_cols(it.rows));
      if (lane == 0) {
        free_item(seq);
        const int h = turn.wide() ? 0 : turn.half();
        ok = mbar_wait(tfull_bar(h), turn.parity(h), s_abort, status) ? 1 : 0;
        if (ok && turn.wide()) ok = mbar_wait(tfull_bar(1), turn.parity(1), s_abort, status) ? 1 : 0;
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) goto done;
      tc_fence_after();
      // this warp's 32 outputs start at fbase
      const bool slim = it.phase == 1 && slim_tile(p.I, it.out);
      int fbase = it.out * (it.phase == 1 ? kFeat1 : kFeat2) + (int)rank * 128 + q * 32, token0 = 0, cols = entry_cols(it.rows);
      if (slim) {   // lanes 0..63: the CTA's 64 outputs of the first half of the tokens, lanes 64..127: of the second half
        fbase = it.out * kFeat1 + (int)rank * 64 + (q & 1) * 32;
        cols >>= 1;
        token0 = (q >> 1) * cols;
      }
      auto run = [&](auto phase, bf16* out, int n_out) {
        constexpr int PH = decltype(phase)::value;
        if (cols <= 64) epilogue_tile<PH, 2>(it, turn, taddr, chunk0, lane, fbase, token0, cols, tile, p.slots, out, n_out, tempty_bar(0), tempty_bar(1));
        else if (cols <= 128) epilogue_tile<PH, 4>(it, turn, taddr, chunk0, lane, fbase, token0, cols, tile, p.slots, out, n_out, tempty_bar(0), tempty_bar(1));
        else epilogue_tile<PH, 8>(it, turn, taddr, chunk0, lane, fbase, token0, cols, tile, p.slots, out, n_out, tempty_bar(0), tempty_bar(1));
      };
      if (it.phase == 1) {
        run(std::integral_constant<int, 1>(), p.act_out, p.I);
        // this warp's part of the intermediate is written: the publisher counts the CTA's share of the tile
        __syncwarp();
        if (lane == 0) mbar_arrive_release(part_bar(seq % kParts));
      } else {
        run(std::integral_constant<int, 2>(), p.yp, p.H);
      }
    }
  }

done:
  if (*s_abort) {
    // give copies and MMAs in flight time to land before shared memory and TMEM go away
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // neither CTA leaves while its peer may still touch its memory or barriers
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

// ---- self-test of the bounded wait ---------------------------------------------------------------
// One CTA waits on a barrier that nothing ever arrives on, with a short cycle limit, through the same
// wait routine the expert kernels use: the wait gives up, records EB_ERR_TIMEOUT and the kernel returns.
__global__ void bounded_wait_probe_kernel(long long limit_cycles, int* status, int* gave_up) {
  __shared__ uint64_t bar;
  __shared__ int s_abort;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    bool ok = mbar_wait(smem_u32(&bar), 0, &s_abort, status, limit_cycles);
    *gave_up = ok ? 0 : 1;
  }
}

// ---- tile list construction: eb_tiles.cuh -----------------------------------------------------
__global__ void __launch_bounds__(1024)
plan_kernel(ModelParams mp, const int32_t* __restrict__ group_off, const int32_t* __restrict__ step_meta, int device, TilePlan out) {
  EB_GRID_DEP_SYNC();
  __shared__ OrderShared sh;
  __shared__ int s_dev_off[EB_MAX_D + 1];
  if (threadIdx.x <= mp.D) s_dev_off[threadIdx.x] = mp.dev_off[threadIdx.x];
  const int g0 = device < 0 ? 0 : step_meta[3 + device];
  const int g1 = device < 0 ? step_meta[1] : step_meta[3 + device + 1];
  const int nl = step_meta[2];
  __syncthreads();
  auto item = [&](int i) {
    const int g = group_at(mp, s_dev_off, nl, device, g0, i);
    int head, n_slots;
    if (merged_class(mp, s_dev_off, nl, device, i, group_off, &head, &n_slots)) {
      // the class's tiles sit at its first position
      const int tiles = i == head ? (n_slots + kMergeSlots - 1) / kMergeSlots : 0;
      return Position{g, n_slots, tiles, cost_class(tiles, merged_cols(min(n_slots, kMergeSlots)))};
    }
    const int rows = group_off[g + 1] - group_off[g], tiles = group_tiles(rows);
    return Position{g, -1, tiles, cost_class(tiles, group_cols(rows))};
  };
  order_tiles(g1 - g0, nl, device, g0, item, out, sh);
}

__global__ void __launch_bounds__(256)
fill_kernel(ModelParams mp, const int32_t* __restrict__ group_off, const int32_t* __restrict__ group_w, TileList list) {
  EB_GRID_DEP_SYNC();
  extern __shared__ int s_pref[];
  fill_tiles(mp, group_off, group_w, list, s_pref, blockIdx.x, gridDim.x);
}

// ---- host side ---------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static const EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return (EncodeTiledFn)p;
  }();
  return fn;
}

// bf16 tensor [d2][d1][d0] (d0 innermost), box {b0, b1, 1}, 128-byte swizzle, zero fill out of bounds
bool make_map(CUtensorMap* m, const void* ptr, uint64_t d0, uint64_t d1, uint64_t d2, uint32_t b0, uint32_t b1) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {d0, d1, d2};
  cuuint64_t strides[2] = {d0 * 2, d0 * d1 * 2};
  cuuint32_t box[3] = {b0, b1, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  int rank = d2 > 0 ? 3 : 2;
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

cudaError_t launch_ffn(eb_ctx* c, cudaStream_t st, const FfnParams& p) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c->pair_grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  ++g_ebi_launches;
  return cudaLaunchKernelEx(&cfg, ffn_kernel, p);
}

}  // namespace

eb_status ebi_selftest_wait(eb_ctx* c, cudaStream_t st, long long limit_cycles, int* d_gave_up) {
  bounded_wait_probe_kernel<<<1, 32, 0, st>>>(limit_cycles, c->d_status, d_gave_up);
  EB_LAUNCH_CHECK(c, "bounded wait probe");
  return EB_OK;
}

eb_status ebi_ffn_bind(eb_ctx* c) {
  if (eb_status ds = ebi_check_device(c)) return ds;
  const eb_config& g = c->cfg;
  const uint64_t nw = (uint64_t)g.L * (g.E + g.S);
  // weight tiles: boxes of 128 rows x one k-block, of 64 rows for slim tiles
  if (!make_map(&c->tm_gate, c->w_gate, g.H, g.I, nw, BK, 128) || !make_map(&c->tm_up, c->w_up, g.H, g.I, nw, BK, 128) ||
      !make_map(&c->tm_down, c->w_down, g.I, g.H, nw, BK, 128) || !make_map(&c->tm_gate64, c->w_gate, g.H, g.I, nw, BK, 64) ||
      !make_map(&c->tm_up64, c->w_up, g.H, g.I, nw, BK, 64))
    return ebi_fail(c, EB_ERR_CUDA, "cuTensorMapEncodeTiled failed for the weights");
  // per context: function attributes and cluster occupancy belong to the current device
  cudaError_t e = cudaFuncSetAttribute(ffn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
  if (e != cudaSuccess) return ebi_check_cuda(c, e, "cudaFuncSetAttribute");
  // how many 2-CTA clusters of this kernel the device can hold at once (one CTA per SM)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (c->num_sms / 2));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  e = cudaOccupancyMaxActiveClusters(&clusters, ffn_kernel, &cfg);
  if (e != cudaSuccess || clusters < 1) {
    cudaGetLastError();
    return ebi_fail(c, EB_ERR_CUDA, "the device cannot hold a 2-CTA cluster of the expert kernel");
  }
  c->pair_grid = 2 * (clusters < c->num_sms / 2 ? clusters : c->num_sms / 2);
  return EB_OK;
}

eb_status ebi_ffn_run(eb_ctx* c, cudaStream_t st, const void* xp, const int32_t* group_off, const int32_t* group_w,
                      const int32_t* step_meta, void* yp, int32_t device, bool planned) {
  if (!xp || !group_off || !group_w || !step_meta || !yp) return ebi_fail(c, EB_ERR_INVALID_ARG, "null pointer");
  if (eb_status ds = ebi_check_device(c)) return ds;
  if (!ebi_aligned16(xp) || !ebi_aligned16(yp)) return ebi_fail(c, EB_ERR_INVALID_ARG, "xp / yp must be 16-byte aligned");
  if (!c->w_gate) return ebi_fail(c, EB_ERR_INVALID_ARG, "weights not bound");
  if (!c->ws) return ebi_fail(c, EB_ERR_WORKSPACE, "no workspace set");
  const eb_config& g = c->cfg;
  const int rows = ebi_rows_cap(c);
  // token-row boxes of 128 / 64 / 32 / 16 / 8 rows x one k-block, over the permuted rows and over the intermediate
  FfnParams p;
  const int box_rows[5] = {128, 64, 32, 16, 8};
  for (int i = 0; i < 5; ++i)
    if (!make_map(&p.xp.box[i], xp, g.H, rows, 0, BK, box_rows[i]) || !make_map(&p.act.box[i], c->act, g.I, rows, 0, BK, box_rows[i]))
      return ebi_fail(c, EB_ERR_CUDA, "cuTensorMapEncodeTiled failed for the activations");
  p.gate = c->tm_gate;
  p.up = c->tm_up;
  p.down = c->tm_down;
  p.gate64 = c->tm_gate64;
  p.up64 = c->tm_up64;
  p.work = (const Tile*)c->work;
  p.slots = c->slots;
  p.work_count = c->work_count;
  p.next = c->work_count + 6;
  p.ready = c->tile_ready;
  p.act_out = c->act;
  p.yp = (bf16*)yp;
  p.H = g.H;
  p.I = g.I;
  p.status = c->d_status;
  if (!planned) {
    {
      KernelTimer timer(c, EBK_FFN_PLAN, st);
      EB_LAUNCH(c, "expert_ffn", ebi_launch(plan_kernel, dim3(1), dim3(1024), 0, st, c->mp, group_off, step_meta, (int)device, tile_plan_of(c)));
    }
    KernelTimer timer(c, EBK_FFN_FILL, st);
    EB_LAUNCH(c, "expert_ffn", ebi_launch(fill_kernel, dim3(c->num_sms), dim3(256), sizeof(int) * (size_t)(ebi_groups_cap(c) + 1), st, c->mp,
                                          group_off, group_w, tile_list_of(c)));
  }
  if (!c->timing) {
    p.part = 0;
    EB_LAUNCH(c, "expert_ffn", launch_ffn(c, st, p));
  } else {   // the same tiles in two launches, so that each phase gets a time of its own
    {
      KernelTimer timer(c, EBK_FFN_GATEUP, st);
      p.part = 1;
      EB_LAUNCH(c, "expert_ffn", launch_ffn(c, st, p));
    }
    KernelTimer timer(c, EBK_FFN_DOWN, st);
    p.part = 2;
    EB_LAUNCH(c, "expert_ffn", launch_ffn(c, st, p));
  }
  EB_LAUNCH_CHECK(c, "expert_ffn");
  return EB_OK;
}
