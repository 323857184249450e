// tcgen05 executor for the Ozaki slice-pair products (Sec. "Ozaki Scheme", Fig. 2).
//
// The digits are small integers (|d| <= 127 for the truncated beta = 7 digits,
// <= 128 for the nearest beta = 8 digits), exactly representable in bfloat16,
// so the slice-pair products run on the 5th-generation tensor cores
// (tcgen05.mma kind::f16, bf16 x bf16 -> fp32 in tensor memory). The nearest
// digits of the E4M3 mode (beta = 5, |d| <= 16) are exact E4M3 values and run
// on kind::f8f6f4 at twice the rate, with the same shared-memory layout in
// bytes (a 128-byte swizzle row holds 128 of them instead of 64). An fp32 sum
// of such products is exact while every partial sum stays at most 2^24 in
// magnitude; the K loop is therefore cut into chunks of 1024 (beta = 7 and 8:
// 1024 * 128^2 = 2^24) or 8192 (beta = 5, where 65536 * 16^2 = 2^24 would do) K
// elements. Each chunk lands in one of two TMEM accumulators; while the tensor
// core fills the other, eight epilogue warps drain the finished one into exact
// int32 sums in registers.
//
// A product runs as two kernels:
//   ozaki_tc_kernel      the integer part. A program of slice-pair steps, cut
//                        into segments, is run for every output tile; the
//                        exact sum of a segment is added, times the segment's
//                        power-of-two weights, to the tile's int64 group sums
//                        in an L2-resident area (red.global.add.u64: nothing
//                        comes back). Integer adds commute, so a tile's work
//                        may be shared by any number of CTAs.
//   ozaki_finish_kernel  the float64 part, spread over the whole GPU: the
//                        group sums rounded to float64 in the order of the
//                        definition, unscaled, the update applied and both
//                        triangles written in full lines; the area is zeroed
//                        behind the reads for the next product.
// In the product kernel's epilogue the output step would leave one CTA alone with
// its 128 x 256 part of a tile for 60-75 us while its tensor core waits: at n =
// 256 (one tile) 85 of a product's 95 us, where the two kernels take 16.
// Up to G consecutive levels (G = 4 for beta 7 and 5, 3 for beta 8) form an
// exact group; one or two groups are one exact integer, rounded once, and
// three or more are added in float64 from L = s+1 down to 2 -- the operation
// sequence of the definition, so the float64 result is bit-for-bit the one the
// IMMA executor and the oracle produce.
//
// CTA layout of the product kernel (320 threads, one CTA per SM):
//   warp 0      TMA producer: A tile 128 x 64 and B tile BN x 64 bf16 per K
//               atom, 128-byte swizzle, into a shared-memory ring
//   warp 1      TMEM owner and MMA issuer (one thread): 4 MMAs of K = 16 per
//               atom, commits free the stage and publish finished chunks
//   warps 2..9  epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31 (one output
//               row per thread) and half of the BN columns
// In symmetric mode only tiles holding some element with row <= column run;
// each element with row <= column is computed and written once, and mirrored.
//
// Every mbarrier wait is bounded by a %globaltimer deadline; on expiry the CTA
// raises an error flag, drains what it has in flight (bounded again), frees
// its TMEM and returns.

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>

#include "dmp_internal.cuh"
#include "tile_order.h"

namespace dmp {

namespace {

constexpr int TC_BM = 128;
constexpr int TC_BK = 64;       // bf16 elements per K block: one 128-byte swizzle row
constexpr int TC_ROW_BYTES = 128;  // bytes of one K block row (the swizzle atom width)
constexpr int TC_MMA_PER_ATOM = 4;  // MMAs per K block: 32 bytes of K each (16 bf16 or 32 e4m3)
constexpr int TC_THREADS = 320;
constexpr int TC_EPI_WARPS = 8;
constexpr int kTileRing = 4;  // WALK 2: tile indices the producer may announce ahead

// PAIR: a cluster of two CTAs computes a 256 x BN tile with tcgen05.mma.cta_group::2;
// each CTA stages its own 128 rows of A and half of the BN rows of B, and its
// TMEM receives its 128 output rows with all BN columns.
// A stage holds one K atom (a 128-byte row) of each operand. The copies into the
// SM bound the kernel: an atom of the pair kernel takes 646 clocks (51 bytes per
// clock and SM, at any size and hit rate) against 512 of its MMAs. The ring is
// cut fine so that most of it is in flight (seven stages of one atom: a product
// of n = 8192, s = 5, pairs one by one, 3.69 ms; three of two atoms 3.88). Sharing
// the A rows of two pairs by TMA multicast (a quarter fewer bytes from L2, the
// same into the SMs) leaves the clocks per atom as they are.
template <int BN, bool PAIR = false, bool F8 = false>
struct TcCfg {
  static constexpr int ATOM_K = F8 ? 128 : TC_BK;  // K elements per atom
  static constexpr int A_BYTES = TC_BM * TC_ROW_BYTES;
  static constexpr int B_BYTES = (PAIR ? BN / 2 : BN) * TC_ROW_BYTES;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = PAIR ? 7 : (BN <= 128 ? 6 : 4);
  static constexpr int TMEM_COLS = 2 * BN;      // two fp32 chunk accumulators
  static constexpr int COLS = BN / 2;           // columns per epilogue thread
  static constexpr int BAR_BYTES = 256;
  static constexpr int SMEM = STAGES * STAGE_BYTES + BAR_BYTES + 1024;  // + alignment slack
  static constexpr int BM = PAIR ? 2 * TC_BM : TC_BM;  // rows of a (pair) tile
  static constexpr int RANKS = PAIR ? 2 : 1;
  static constexpr int PART = TC_BM * BN;       // elements of one CTA's part of a tile
};

// The program of one output tile: steps (the product of plane a of A with
// plane b of B over the whole K) in segments. A segment's exact sum goes, times
// w[i], into the group sums g0 + i.
constexpr int kMaxSegs = 32;
constexpr int kMaxSteps = 96;
constexpr int kMaxLaunchTiles = 160;  // single-matrix launches

struct TcSeg {
  int step0, nsteps;
  int g0;
  long long w[3];
};

struct TcProgram {
  int nsegs;
  int ng;       // group sums per element
  TcSeg seg[kMaxSegs];
  unsigned char pa[kMaxSteps], pb[kMaxSteps];  // plane indices of the steps
};

struct TcParams {
  int s, beta, KT, CH;
  int tile0, ntiles;  // this launch's tiles: tile0 .. tile0 + ntiles - 1
  int nwhole;         // tiles (of ntiles) walked whole, round robin; the rest are split over all CTAs (CTA pairs)
  int units;          // fp32 chunks per tile (split launches: one matrix, every tile alike)
  // the first heads * head_len units of each split tile in `heads` equal ranges, one CTA (CTA pair) each; the
  // other units of all split tiles in one sequence, evenly cut over the other CTAs
  int heads, head_len;
  int group;        // levels combined exactly per int64 group: 4 (beta 7, 5) or 3 (beta 8)
  double gscale[3];   // three groups: the weights 2^(-beta (s + 1 - group g)) of their sums
  long long* area;  // group sums of the launch's tiles: [tile][CTA rank][group][PART]
  int64_t m, n;
  int64_t rows_a, rows_b;  // padded rows per digit plane
  int sym;
  int column_bits;  // of the words in `at`
  const int32_t* ea;
  const int32_t* eb;
  EpiArgs epi;
  const int* done;
  int* err;
  unsigned long long timeout_ns;
  int stall_test;  // withhold each CTA's first stage (the bounded-wait test; see dmp_test_stall_next_product)
  int* tile_counter;  // WALK 2: next tile to take (zeroed before the launch)
  // grouped mode (batched purification): tiles of many matrices in one launch
  const BatchMat* mats;  // nullptr: the single matrix above
  const int4* tiles;     // {matrix, bi, bj, 0}
  int phase;             // 0: X2 = P P;  1: P' = update(P, X2, P X2)
  int cur;               // the iterate is mats[.].buf[cur]
  TcProgram prog;
  // single-matrix launches: row and column block of each of the launch's tiles
  // (a table: finding a tile's place in the order by counting took the finish
  // kernel a thousand instructions per warp), packed with column_bits bits
  uint32_t at[kMaxLaunchTiles];
};

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// one lane of the (converged) warp, always the same
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok));
  return ok != 0;
}
__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(tm), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void tma_prefetch(const CUtensorMap* tm) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(tm) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// ---- the CTA pair (cluster of two, cta_group::2)
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// the shared::cluster address of the same object in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, "
      "p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// arrive on a barrier of either CTA of the pair (a shared::cluster address).
// Used only to hand a TMEM buffer back to the MMA issuer: the loads from it
// have completed (tcgen05.wait::ld) and are ordered before the arrive by
// tcgen05.fence::before_thread_sync, and no memory this thread wrote is passed
// on through the barrier. The arrive therefore keeps the default CTA-scope
// release: a cluster-scope release adds a fence on every drained chunk that
// waits for the thread's outstanding memory operations.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// TMA load into this CTA's shared memory that signals `bar`, which may be the peer's
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, "
      "%4}], [%2];" ::"r"(dst),
      "l"(tm), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void umma_e4m3(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_e4m3_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// one MMA of the 256-row pair tile: A rows from both CTAs, B halves from both
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrive on `bar` in both CTAs of the pair when the MMAs issued so far complete
__device__ __forceinline__ void umma_commit_pair_both(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"(static_cast<unsigned short>(3))
      : "memory");
}
__device__ __forceinline__ void umma_commit_pair_self(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// L2 evict-last policy for the group sums: touched once per segment while
// gigabytes of operand tiles stream through L2
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
// 64-bit integer add performed at L2 (no value returned, so no round trip):
// two's complement, so it adds signed values exactly
__device__ __forceinline__ void red_add_keep(void* p, long long v, uint64_t pol) {
  asm volatile("red.global.add.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(p), "l"(v), "l"(pol) : "memory");
}

// RN(x) 2^e as a double for the signed 96-bit integer x = (w2:w1:w0), rounded to
// nearest even: the value of the float64 expression in which x is the exact sum
// of its groups. Integer operations only: float64 conversions, multiplies and
// adds run on this GPU's narrow FP64 pipe (two lanes per clock and SM), which
// bound the finish kernel at 83 % of its issue rate when it used them.
__device__ __forceinline__ double round_words(uint32_t w0, uint32_t w1, uint32_t w2, int e) {
  const uint32_t neg = static_cast<uint32_t>(static_cast<int32_t>(w2) >> 31);  // all ones when negative
  // magnitude: (x ^ neg) - neg
  uint32_t a0 = w0 ^ neg, a1 = w1 ^ neg, a2 = w2 ^ neg;
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.u32 %2, %2, 0;"
      : "+r"(a0), "+r"(a1), "+r"(a2)
      : "r"(neg & 1u));
  // leading zeros, then the magnitude shifted so that its top bit is bit 95
  int lz = 0;
  if (a2 == 0) {
    a2 = a1;
    a1 = a0;
    a0 = 0;
    lz = 32;
    if (a2 == 0) {
      a2 = a1;
      a1 = 0;
      lz = 64;
      if (a2 == 0) return 0.0;
    }
  }
  const int z = __clz(static_cast<int>(a2));
  lz += z;
  a2 = __funnelshift_l(a1, a2, z);
  a1 = __funnelshift_l(a0, a1, z);
  a0 <<= z;
  // 53 bits: a2 and the top 21 bits of a1; the rest rounds to nearest even
  const uint32_t rest = (a1 << 21) | (a0 != 0 ? 1u : 0u);
  uint32_t lo = (a2 << 21) | (a1 >> 11), hi = a2 >> 11;
  const uint32_t up = (rest > 0x80000000u || (rest == 0x80000000u && (lo & 1u))) ? 1u : 0u;
  const int E = 95 - lz + e + 1023;  // biased exponent before rounding
  // the leading one (bit 20 of hi) adds one to the exponent field, and so does a carry out of the fraction
  hi += static_cast<uint32_t>(E - 1) << 20;
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(lo), "+r"(hi) : "r"(up));
  if (E < 1 || E > 2045) {
    // outside the normal range: the rounded integer scaled by ldexp
    uint32_t l0 = (a2 << 21) | (a1 >> 11), h0 = (a2 >> 11) + (static_cast<uint32_t>(95 - lz + 1022) << 20);
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(l0), "+r"(h0) : "r"(up));
    const double v = ldexp(__hiloint2double(static_cast<int>(h0), static_cast<int>(l0)), e);
    return neg ? -v : v;
  }
  return __hiloint2double(static_cast<int>(hi | (neg & 0x80000000u)), static_cast<int>(lo));
}

// The same for a signed 64-bit integer x = (w1:w0), without branches, so that
// the elements of a thread overlap. `slow` is raised (and the value to be taken
// from round_words) when the result is not a normal number.
__device__ __forceinline__ double round_fast2(uint32_t w0, uint32_t w1, int e, bool& slow) {
  const uint32_t neg = static_cast<uint32_t>(static_cast<int32_t>(w1) >> 31);
  uint32_t a0 = w0 ^ neg, a1 = w1 ^ neg;
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(a0), "+r"(a1) : "r"(neg & 1u));
  const bool small = a1 == 0;
  a1 = small ? a0 : a1;
  a0 = small ? 0u : a0;
  const int z = __clz(static_cast<int>(a1));  // 32 for zero
  const bool zero = a1 == 0;
  a1 = __funnelshift_l(a0, a1, z);
  a0 <<= z & 31;
  uint32_t lo = (a1 << 21) | (a0 >> 11), hi = a1 >> 11;
  // up on more than half, or on half with an odd last bit
  const uint32_t up = ((a0 & 0x7ffu) + (lo & 1u)) > 0x400u ? 1u : 0u;
  const int E = (small ? 31 : 63) - z + e + 1023;  // biased exponent before rounding
  slow |= !zero && static_cast<uint32_t>(E - 1) > 2044u;
  hi += static_cast<uint32_t>(E - 1) << 20;
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(lo), "+r"(hi) : "r"(up));
  hi |= neg & 0x80000000u;
  return __hiloint2double(zero ? 0 : static_cast<int>(hi), zero ? 0 : static_cast<int>(lo));
}

// x 2^e for a finite double: exponent arithmetic when the result stays normal,
// ldexp otherwise (identical results: scaling by a power of two is exact).
__device__ __forceinline__ double scale_pow2(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int E = static_cast<int>((b >> 52) & 0x7ff);
  const int En = E + e;
  if (E != 0 && E != 0x7ff && En > 0 && En < 0x7ff) return __longlong_as_double(b + (static_cast<long long>(e) << 52));
  return ldexp(x, e);
}

// Shared-memory matrix descriptor: K-major operand tile, rows of 128 bytes,
// 128-byte swizzle, 8-row groups 1024 bytes apart (tile base 1024-aligned).
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr >> 4) & 0x3FFFu);  // start address
  d |= static_cast<uint64_t>(1) << 16;                  // leading byte offset (unused for this layout)
  d |= static_cast<uint64_t>(1024 >> 4) << 32;          // stride byte offset: 8 rows
  d |= static_cast<uint64_t>(1) << 46;                  // descriptor version
  d |= static_cast<uint64_t>(2) << 61;                  // 128-byte swizzle
  return d;
}
// Instruction descriptor, kind::f16: fp32 D, bf16 A and B, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(M >> 4) << 24);
}
// Instruction descriptor, kind::f8f6f4: fp32 D, E4M3 A and B (format 0), both K-major.
__host__ __device__ constexpr uint32_t idesc_e4m3(int M, int N) {
  return (1u << 4) | (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}

// bounded wait; false on timeout or when another role aborted. CLUSTER: the
// barrier also receives arrivals from the peer CTA (acquire at cluster scope).
template <bool CLUSTER = false>
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                         const TcParams& p) {
  auto try_once = [&]() { return CLUSTER ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity); };
  if (try_once()) return true;
  const uint64_t deadline = globaltimer() + p.timeout_ns;
  for (uint32_t it = 1;; ++it) {
    if (try_once()) return true;
    if ((it & 255u) == 0) {
      if (*abort_flag) return false;
      if (globaltimer() > deadline) {
        *abort_flag = 1;
        if (p.err != nullptr) atomicExch(p.err, 1);
        return false;
      }
    }
  }
}
// Where one CTA's part of an output tile lies and what feeds it.
struct Job {
  const CUtensorMap* ta;
  const CUtensorMap* tb;
  int64_t m0, n0, rows_a, rows_b;
  int KT;
  bool skip;
};

// tile: counted from the launch's first (tile0).
// PAIR: tile is a 256-row pair tile and this CTA (rank 0 or 1) takes rows
// 128 rank .. 128 rank + 127 of it.
template <int BN, bool PAIR>
__device__ __forceinline__ Job job_of(const TcParams& p, const CUtensorMap* tmA, const CUtensorMap* tmB, int tile,
                                      uint32_t rank) {
  constexpr int BM = TcCfg<BN, PAIR>::BM;
  Job j;
  if (p.mats == nullptr) {
    j.ta = tmA;
    j.tb = tmB;
    const TileAt at = unpack_tile(p.at[tile], p.column_bits);
    j.m0 = static_cast<int64_t>(at.bi) * BM + TC_BM * static_cast<int64_t>(rank);
    j.n0 = static_cast<int64_t>(at.bj) * BN;
    j.rows_a = p.rows_a;
    j.rows_b = p.rows_b;
    j.KT = p.KT;
    j.skip = false;
    return j;
  }
  const int4 t = p.tiles[p.tile0 + tile];
  const BatchMat& M = p.mats[t.x];
  j.m0 = static_cast<int64_t>(t.y) * BM + TC_BM * static_cast<int64_t>(rank);
  j.n0 = static_cast<int64_t>(t.z) * BN;
  j.rows_a = M.n_pad;
  j.rows_b = M.n_pad;
  j.KT = static_cast<int>(M.k_pad / (p.beta == 5 ? 128 : TC_BK));  // K atoms of 128 bytes
  j.skip = M.state->done != 0;
  j.ta = &M.tmPa;
  j.tb = p.phase == 0 ? &M.tmPb : &M.tmXb;
  return j;
}

// Four consecutive doubles or int64 group sums, in 16-byte pieces when the
// address allows (`vec`), else one by one at immediate offsets.
__device__ __forceinline__ void load4(double (&v)[4], const double* a, bool vec) {
  if (vec) {
    const double2 x = reinterpret_cast<const double2*>(a)[0], y = reinterpret_cast<const double2*>(a)[1];
    v[0] = x.x, v[1] = x.y, v[2] = y.x, v[3] = y.y;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = a[i];
  }
}
__device__ __forceinline__ void store4(double* a, const double (&v)[4], bool vec) {
  if (vec) {
    reinterpret_cast<double2*>(a)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(a)[1] = make_double2(v[2], v[3]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = v[i];
  }
}

// The float64 part of a product, one CTA per 32 x 32 block of a tile, four rows
// of a column per thread and pass. The group sums lie as [column][row], P and
// P^2 are exactly symmetric (read at (column, row)) and the mirrored elements
// are four in a row too, so every array costs a thread one address and 16-byte
// accesses; the row-major elements go through shared memory for the same
// reason. n = 4096: 40 us (with the update 60, 45 of them the FP64 pipe's)
// beside 470 of products, n = 1024: 6 (9) beside 29.
// (On two further warps of the next wave's product kernel it costs 3 % of the
// whole: 200 us per wave of 76 tiles on so few threads, and the shared memory of
// a seventh stage.)
// OUT: what becomes of an element. NG: group sums per element (0: EPI_LEVELS).
constexpr int FIN_THREADS = 128;
enum { OUT_STORE = 0, OUT_UPDATE = 1, OUT_CHEB = 2 };  // EPI_STORE and EPI_SYM_STORE, EPI_PM_UPDATE, EPI_CHEB

template <int BN, bool PAIR, int OUT, int NG>
__global__ void __launch_bounds__(FIN_THREADS)
ozaki_finish_kernel(const __grid_constant__ TcParams p) {
  chain_wait();
  chain_next();
  constexpr bool UPD = OUT == OUT_UPDATE, CHEB = OUT == OUT_CHEB;
  __shared__ double trans[32][33];
  using Cfg = TcCfg<BN, PAIR>;
  constexpr int SR = Cfg::BM / 32, SC = BN / 32;
  constexpr int LINES = FIN_THREADS / 8, PASSES = 32 / LINES;  // lines of a block per pass
  const int q4 = 4 * (threadIdx.x & 7), line0 = threadIdx.x >> 3;  // four entries of lines line0, line0 + LINES, ..
  const bool sym = p.sym != 0;
  const int e_sum = -p.beta * (p.s + 1);

  const int tile = blockIdx.x / (SR * SC);
  const int sub = blockIdx.x % (SR * SC);
  const int sr = sub % SR, sc = sub / SR;
  const int rank = sr / 4;
  const int h = 32 * sc / Cfg::COLS;
  const int e = 4 * h + ((sr + 2) & 3);  // the epilogue warp that owns these rows and columns

  // The group sums first: their place follows from the block alone, so they are
  // on their way while the batch's tile, matrix and state are looked up one after
  // the other, and so does the check of the done flag (152 tiles of a batch: 42 us,
  // with the update 65; 107 and 123 with the loads after the check).
  constexpr int G = NG == 0 ? 1 : NG;
  long long* part0 = p.area + (static_cast<int64_t>(tile) * Cfg::RANKS + rank) * (NG == 0 ? p.prog.ng : NG) * Cfg::PART +
                     (e * (Cfg::COLS * 32) + (32 * sc - h * Cfg::COLS + line0) * 32 + q4);
  long long T[PASSES][G][4];
#pragma unroll
  for (int pass = 0; pass < PASSES; ++pass) {
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      const longlong2* a = reinterpret_cast<const longlong2*>(part0 + g * Cfg::PART + pass * (LINES * 32));
      const longlong2 x = a[0], y = a[1];
      T[pass][g][0] = x.x, T[pass][g][1] = x.y, T[pass][g][2] = y.x, T[pass][g][3] = y.y;
    }
  }

  // the tile's place and its output step
  int done = p.done != nullptr ? *p.done : 0;
  int m0, n0, m = static_cast<int>(p.m), n = static_cast<int>(p.n);
  const int32_t* ea = p.ea;
  const int32_t* eb = p.eb;
  EpiArgs epi = p.epi;
  if (p.mats == nullptr) {
    const TileAt at = unpack_tile(p.at[tile], p.column_bits);
    m0 = at.bi * Cfg::BM;
    n0 = at.bj * BN;
  } else {
    const int4 t = p.tiles[p.tile0 + tile];
    const BatchMat& M = p.mats[t.x];
    done = M.state->done;
    m0 = t.y * Cfg::BM;
    n0 = t.z * BN;
    m = n = static_cast<int>(M.n);
    ea = M.expsP;
    epi.state = M.state;
    if (!UPD) {
      eb = M.expsP;
      epi.C = M.X2;
      epi.ldc = M.n;
    } else {
      eb = M.expsX;
      epi.P = M.buf[p.cur];
      epi.ldp = p.cur == 0 ? M.ldp : M.n;
      epi.X2 = M.X2;
      epi.ldx = M.n;
      epi.C = M.buf[1 - p.cur];
      epi.ldc = p.cur == 0 ? M.n : M.ldp;
    }
  }
  const int r0 = m0 + 32 * sr, c0 = n0 + 32 * sc;
  const int r = r0 + q4;  // this thread's first row
  // nothing of this block is written: outside the matrix, or below the diagonal
  const bool none = r0 >= m || c0 >= n || (sym && r0 > c0 + 31);
  const bool vec = (epi.ldc & 1) == 0 && (reinterpret_cast<uintptr_t>(epi.C) & 15) == 0;

  if constexpr (NG == 0) {
    if (done) return;
    // test hook: group g holds the exact sum of level g + 2
    for (int pass = 0; pass < PASSES; ++pass) {
      const int c = c0 + line0 + LINES * pass;
      for (int g = 0; g < p.prog.ng; ++g) {
        long long* part = part0 + g * Cfg::PART + pass * (LINES * 32);
        for (int t = 0; t < 4; ++t) {
          if (r + t < m && c < n)
            epi.levels[(static_cast<int64_t>(g) * m + r + t) * n + c] = static_cast<int32_t>(part[t]);
          part[t] = 0;
        }
      }
    }
    return;
  }

  // the exponents beside the check, the rest after it; every load of the block
  // before the first store, so that a thread waits for few rounds of latencies
  double pv[PASSES][4], xv[PASSES][4];
  int32_t ec[PASSES];
  int4 er4 = make_int4(0, 0, 0, 0);
  if (r < m) er4 = *reinterpret_cast<const int4*>(ea + r);  // (the exponent arrays are padded to 256 rows)
  const int32_t er[4] = {er4.x, er4.y, er4.z, er4.w};
#pragma unroll
  for (int pass = 0; pass < PASSES; ++pass) {
    const int c = c0 + line0 + LINES * pass;
    ec[pass] = c < n ? eb[c] : 0;
  }
  const double wa = UPD ? epi.state->alpha : 0.0;
  const double w2 = UPD ? epi.state->b2 : 0.0;
  const double w3 = UPD ? epi.state->b3 : 0.0;
  const double coef = CHEB && epi.acc != nullptr ? *epi.coef : 0.0;
  if (done) return;
  // the update's P and P^2; the recurrence's term before and its running sum
  const bool two = UPD || (CHEB && epi.acc != nullptr), one = UPD || (CHEB && epi.P != nullptr);
  const double* xbase = CHEB ? epi.acc : epi.X2;
  const int64_t ldx = CHEB ? epi.ldacc : epi.ldx;
  const double* pp = one ? epi.P + (c0 + line0) * epi.ldp + r : nullptr;
  const double* xp = two ? xbase + (c0 + line0) * ldx + r : nullptr;
  const bool vecp = one && (epi.ldp & 1) == 0 && (reinterpret_cast<uintptr_t>(epi.P) & 15) == 0;
  const bool vecx = two && (ldx & 1) == 0 && (reinterpret_cast<uintptr_t>(xbase) & 15) == 0;
#pragma unroll
  for (int pass = 0; pass < PASSES; ++pass) {
    const int c = c0 + line0 + LINES * pass;
    if (UPD || CHEB) {
      // the rows of this column that are written: inside the matrix, and not below the diagonal
      const int rows = c < n ? min(sym ? c + 1 : m, m) - r : 0;
      const double* pc = pp + static_cast<int64_t>(LINES * pass) * epi.ldp;
      const double* xc = xp + static_cast<int64_t>(LINES * pass) * ldx;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        // no term before: the identity
        pv[pass][t] = CHEB && epi.P == nullptr && r + t == c ? 1.0 : 0.0;
        xv[pass][t] = 0.0;
      }
      if (rows >= 4) {
        if (one) load4(pv[pass], pc, vecp);
        if (two) load4(xv[pass], xc, vecx);
      } else {
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          if (t < rows) {
            if (one) pv[pass][t] = pc[t];
            if (two) xv[pass][t] = xc[t];
          }
        }
      }
    }
  }
#pragma unroll
  for (int pass = 0; pass < PASSES; ++pass) {
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      longlong2* a = reinterpret_cast<longlong2*>(part0 + g * Cfg::PART + pass * (LINES * 32));
      a[0] = a[1] = make_longlong2(0, 0);
    }
  }
  if (none) return;
#pragma unroll
  for (int pass = 0; pass < PASSES; ++pass) {
    const int line = line0 + LINES * pass;
    const int c = c0 + line;
    const int rows = c < n ? min(sym ? c + 1 : m, m) - r : 0;  // t < rows
    double v[4];
    // one or two groups: the exact integer T_1 2^(beta G) + T_0 rounded once and
    // scaled by 2^(-beta (s+1)) (exact); three: the groups scaled and added in
    // float64 from the smallest up
    bool slow = ec[pass] == kBadExp;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      slow |= er[t] == kBadExp;
      if (NG == 1) {
        v[t] = round_fast2(static_cast<uint32_t>(T[pass][0][t]), static_cast<uint32_t>(T[pass][0][t] >> 32),
                           er[t] + ec[pass] + e_sum, slow);
      } else {
        slow = true;
      }
    }
    if (NG != 1 || slow) {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int ee = er[t] + ec[pass];
        const long long t0 = T[pass][0][t], t1 = T[pass][NG > 1 ? 1 : 0][t], t2 = T[pass][NG > 2 ? 2 : 0][t];
        const uint32_t l0 = static_cast<uint32_t>(t0), h0 = static_cast<uint32_t>(t0 >> 32);
        const uint32_t x0 = static_cast<uint32_t>(static_cast<int32_t>(h0) >> 31);
        if (NG == 1) {
          v[t] = round_words(l0, h0, x0, ee + e_sum);
        } else if (NG == 2) {
          // T_1 shifted by beta G = 20 .. 28 bits, plus T_0 (|T| < 2^53 each)
          const int sh = p.beta * p.group;
          const uint32_t l1 = static_cast<uint32_t>(t1), h1 = static_cast<uint32_t>(t1 >> 32);
          const uint32_t x1 = static_cast<uint32_t>(static_cast<int32_t>(h1) >> 31);
          uint32_t w0 = l1 << sh, w1 = __funnelshift_l(l1, h1, sh), w2s = __funnelshift_l(h1, x1, sh);
          asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
              : "+r"(w0), "+r"(w1), "+r"(w2s)
              : "r"(l0), "r"(h0), "r"(x0));
          v[t] = round_words(w0, w1, w2s, ee + e_sum);
        } else {
          const double d0 = static_cast<double>(t0) * p.gscale[0];
          const double d1 = d0 + static_cast<double>(t1) * p.gscale[1];
          v[t] = scale_pow2(d1 + static_cast<double>(t2) * p.gscale[2], ee);
        }
        if (er[t] == kBadExp || ec[pass] == kBadExp) v[t] = __longlong_as_double(0x7ff8000000000000ll);
      }
    }
    if (UPD) {
#pragma unroll
      for (int t = 0; t < 4; ++t) v[t] = wa * pv[pass][t] + w2 * xv[pass][t] + w3 * v[t];
    }
    if (CHEB) {
#pragma unroll
      for (int t = 0; t < 4; ++t) v[t] = 2.0 * v[t] - pv[pass][t];
      if (epi.acc != nullptr && rows > 0) {
        // both triangles of the running sum (no other thread reads or writes these elements)
        double* a = epi.acc + c * epi.ldacc + r;
        double* am = epi.acc + r * epi.ldacc + c;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          if (t < rows) {
            const double x = xv[pass][t] + coef * v[t];
            a[t] = x;
            am[t * epi.ldacc] = x;
          }
        }
      }
    }
    if (epi.round32 != 0) {
      // stored_value; volatile, so that without the flag the two conversions
      // (FP64 pipe) are branched over instead of being computed and dropped
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float f;
        asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(f) : "d"(v[t]));
        asm volatile("cvt.f64.f32 %0, %1;" : "=d"(v[t]) : "f"(f));
      }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) trans[line][q4 + t] = v[t];
    if (sym && rows > 0) {
      double* mirror = epi.C + c * epi.ldc + r;
      if (rows >= 4) {
        store4(mirror, v, vec);
      } else {
#pragma unroll
        for (int t = 0; t < 3; ++t)
          if (t < rows) mirror[t] = v[t];
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int pass = 0; pass < PASSES; ++pass) {
    // row r0 + line, columns c0 + q4 .. + 3 (symmetric: right of the diagonal)
    const int line = line0 + LINES * pass;
    const int rr = r0 + line, cc = c0 + q4;
    if (rr >= m) continue;
    const int first = sym ? rr + 1 - cc : 0;  // first column of the four that is written
    double* out = epi.C + rr * epi.ldc + cc;
    double v[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) v[t] = trans[q4 + t][line];
    if (first <= 0 && cc + 4 <= n) {
      store4(out, v, vec);
    } else {
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t >= first && cc + t < n) out[t] = v[t];
    }
  }
}

// Persistent: each CTA (CTA pair) walks its share of the launch's tiles. The
// three roles keep their ring and buffer phases across tiles, so the next
// tile's loads and MMAs overlap the current tile's last adds.
//
// PAIR (launched as clusters of two CTAs): the cluster walks 256-row pair
// tiles. Each CTA loads its A rows and its half of the B rows, signalling the
// leader's (rank 0) full barrier; the leader alone issues the cta_group::2
// MMAs and its commits arrive on the stage and accumulator barriers of both
// CTAs; both epilogues release a TMEM buffer on the leader's barrier.
//
// WALK: how the CTAs share the launch's tiles.
//   0  the first p.nwhole tiles whole, round robin; the others (less than one
//      per CTA or CTA pair) are cut into units of one exact fp32 chunk and
//      shared out evenly, in contiguous ranges, over every CTA, so that no
//      last wave is left half empty. The group sums are integers: the result
//      does not depend on the split.
//   2  each CTA takes the next tile from a counter in global memory (the
//      grouped launches of the batched purification, whose tiles differ in
//      work: listed largest first, taken as CTAs free up); the producer takes
//      the tile and passes its index to the MMA and epilogue warps through a
//      small ring in shared memory
template <int BN, bool PAIR, bool F8 = false, int WALK = 0>
__global__ void __launch_bounds__(TC_THREADS, 1)
ozaki_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const __grid_constant__ TcParams p) {
  using Cfg = TcCfg<BN, PAIR, F8>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  uint8_t* barp = smem + Cfg::STAGES * Cfg::STAGE_BYTES;
  const uint32_t bar0 = smem_u32(barp);
  auto full_bar = [&](int st) { return bar0 + 8u * st; };
  auto empty_bar = [&](int st) { return bar0 + 8u * (Cfg::STAGES + st); };
  auto accfull_bar = [&](int b) { return bar0 + 8u * (2 * Cfg::STAGES + b); };
  auto accempty_bar = [&](int b) { return bar0 + 8u * (2 * Cfg::STAGES + 2 + b); };
  const uint32_t drain_bar = bar0 + 8u * (2 * Cfg::STAGES + 4);
  // WALK 2: ring of tile indices from the producer to the MMA and epilogue warps
  auto ring_full = [&](int r) { return bar0 + 8u * (2 * Cfg::STAGES + 5 + r); };
  auto ring_empty = [&](int r) { return bar0 + 8u * (2 * Cfg::STAGES + 5 + kTileRing + r); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(barp + 8 * (2 * Cfg::STAGES + 5 + 2 * kTileRing));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* ring_tile = reinterpret_cast<volatile int*>(tmem_slot + 2);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = PAIR ? cluster_rank() : 0u;
  const bool leader = rank == 0;
  // CTA (or CTA pair) index and count for the persistent tile walk
  const int cta_id = PAIR ? static_cast<int>(blockIdx.x >> 1) : static_cast<int>(blockIdx.x);
  const int cta_stride = PAIR ? static_cast<int>(gridDim.x >> 1) : static_cast<int>(gridDim.x);

  if (threadIdx.x == 0) {
    for (int st = 0; st < Cfg::STAGES; ++st) {
      mbar_init(full_bar(st), 1);
      mbar_init(empty_bar(st), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accfull_bar(b), 1);
      mbar_init(accempty_bar(b), PAIR ? 2 * TC_EPI_WARPS : TC_EPI_WARPS);
    }
    mbar_init(drain_bar, 1);
    if (WALK == 2) {
      for (int r = 0; r < kTileRing; ++r) {
        mbar_init(ring_full(r), 1);
        mbar_init(ring_empty(r), 1 + TC_EPI_WARPS);  // the MMA issuer and every epilogue warp
      }
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0 && p.mats == nullptr) {
    tma_prefetch(&tmA);
    tma_prefetch(&tmB);
  }
  if (warp == 1) {
    if (PAIR) {
      tmem_alloc_pair(smem_u32(tmem_slot), Cfg::TMEM_COLS);  // both CTAs, the same columns
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(tmem_slot), Cfg::TMEM_COLS);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();  // barriers of both CTAs initialised before any remote use
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // the setup above touches no device memory; a set done flag leaves the CTA without tiles
  // (the grouped walk looks at each matrix's own flag)
  chain_wait();
  chain_next();
  const int done = p.done != nullptr ? *p.done : 0;

  const int CHS = p.CH;  // stages per fp32 chunk

  // WALK 0: this CTA's items. Items 0 .. nfull - 1 are whole tiles; after them
  // come the tiles its range [u_begin, u_end) of the split tiles' units meets.
  const int nfull = !done && p.nwhole > cta_id ? (p.nwhole - cta_id - 1) / cta_stride + 1 : 0;
  // (u_end - u_begin units of the sequence of the tiles' units seg_off .. seg_off + seg_len - 1)
  const int nsplit = p.ntiles - p.nwhole;
  const int heads = nsplit * p.heads;
  int64_t u_begin, u_end;
  int seg_off = 0, seg_len = p.units;
  if (cta_id < heads) {
    const int part = cta_id / nsplit;
    seg_off = part * p.head_len;
    seg_len = max(min(p.head_len, p.units - seg_off), 0);
    u_begin = static_cast<int64_t>(cta_id - part * nsplit) * seg_len;
    u_end = u_begin + seg_len;
  } else {
    seg_off = p.heads * p.head_len;
    seg_len = max(p.units - seg_off, 0);
    const int64_t all = static_cast<int64_t>(nsplit) * seg_len;
    u_begin = all * (cta_id - heads) / max(cta_stride - heads, 1);
    u_end = all * (cta_id - heads + 1) / max(cta_stride - heads, 1);
  }
  if (done) u_end = u_begin;
  // item `it`: its tile (counted from tile0) and unit range [u0, u1); false past the last
  auto static_item = [&](int it, int& tile, int& u0, int& u1) __attribute__((always_inline)) -> bool {
    if (it < nfull) {
      tile = cta_id + it * cta_stride;
      u0 = 0;
      u1 = 0x7fffffff;
      return true;
    }
    if (u_begin >= u_end) return false;
    const int tt = static_cast<int>(u_begin / seg_len) + (it - nfull);
    const int64_t base = static_cast<int64_t>(tt) * seg_len;
    if (base >= u_end) return false;
    tile = p.nwhole + tt;
    u0 = seg_off + static_cast<int>(u_begin > base ? u_begin - base : 0);
    u1 = seg_off + static_cast<int>(u_end - base < seg_len ? u_end - base : seg_len);
    return true;
  };

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      // for the abort drain: stages ever armed, and the parity of the phase each
      // was last armed in (that phase completes when its copies have landed)
      uint32_t armed = 0, armed_par = 0;
      bool withheld = false;  // stall test: the first stage has been withheld
      // PAIR: both CTAs' copies complete on the leader's full barrier, which expects both
      const uint32_t full_target0 = PAIR ? map_to_cta(full_bar(0), 0) : full_bar(0);
      const uint32_t expect_bytes = PAIR ? 2u * Cfg::STAGE_BYTES : static_cast<uint32_t>(Cfg::STAGE_BYTES);
      const int b_off = PAIR ? static_cast<int>(rank) * (BN / 2) : 0;  // this CTA's half of the B rows
      // one stage: K atom kt of planes pa of A and pb of B
      auto put_stage = [&](const Job& jb, int pa, int pb, int kt) __attribute__((always_inline)) -> bool {
        if (!wait_bar<PAIR>(empty_bar(stage), phase ^ 1u, abort_flag, p)) return false;
        const int ya = static_cast<int>(pa * jb.rows_a + jb.m0);
        const int yb = static_cast<int>(pb * jb.rows_b + jb.n0) + b_off;
        const uint32_t sa = sbase + stage * Cfg::STAGE_BYTES;
        if (p.stall_test && !withheld) {
          // stall test: neither the expected bytes nor the copies of this CTA's
          // first stage are issued, so its full barrier never completes and
          // the MMA issuer's bounded wait on it runs out (nothing is in
          // flight for this stage; the later stages drain as in any abort)
          withheld = true;
        } else {
          if (PAIR) {
            const uint32_t fb = full_target0 + 8u * stage;
            if (leader) mbar_arrive_expect_tx(full_bar(stage), expect_bytes);
            tma_load_2d_pair(sa, jb.ta, fb, kt * Cfg::ATOM_K, ya);
            tma_load_2d_pair(sa + Cfg::A_BYTES, jb.tb, fb, kt * Cfg::ATOM_K, yb);
          } else {
            mbar_arrive_expect_tx(full_bar(stage), expect_bytes);
            tma_load_2d(sa, jb.ta, full_bar(stage), kt * Cfg::ATOM_K, ya);
            tma_load_2d(sa + Cfg::A_BYTES, jb.tb, full_bar(stage), kt * Cfg::ATOM_K, yb);
          }
          armed |= 1u << stage;
          armed_par = (armed_par & ~(1u << stage)) | (phase << stage);
        }
        if (++stage == Cfg::STAGES) {
          stage = 0;
          phase ^= 1u;
        }
        return true;
      };
      int rslot = 0;
      uint32_t rph = 0;
      for (int it = 0; ok; ++it) {
        int tile = 0, u0 = 0, u1 = 0x7fffffff;
        if constexpr (WALK == 2) {
          // take the next tile from the global counter (skipping finished
          // matrices) and announce it, or -1, to the other warps through the ring
          tile = atomicAdd(p.tile_counter, 1);
          while (tile < p.ntiles && job_of<BN, PAIR>(p, &tmA, &tmB, tile, rank).skip)
            tile = atomicAdd(p.tile_counter, 1);
          if (tile >= p.ntiles) tile = -1;
          if (!wait_bar<false>(ring_empty(rslot), rph ^ 1u, abort_flag, p)) {
            ok = false;
            break;
          }
          ring_tile[rslot] = tile;
          mbar_arrive(ring_full(rslot));  // release: the index is visible to the waiting warps
          if (++rslot == kTileRing) {
            rslot = 0;
            rph ^= 1u;
          }
          if (tile < 0) break;
        } else {
          if (!static_item(it, tile, u0, u1)) break;
        }
        const Job jb = job_of<BN, PAIR>(p, &tmA, &tmB, tile, rank);
        if (jb.skip) continue;
        const int KTS = jb.KT;
        int base = 0;
        for (int g = 0; g < p.prog.nsegs && ok; ++g) {
          const int nkb = p.prog.seg[g].nsteps * KTS;
          const int nch = (nkb + CHS - 1) / CHS;
          const int lo = max(u0 - base, 0), hi = min(u1 - base, nch);
          base += nch;
          if (lo >= hi) continue;
          const int kb1 = min(hi * CHS, nkb);
          int step = p.prog.seg[g].step0 + lo * CHS / KTS;
          int kt = lo * CHS % KTS;
          for (int kb = lo * CHS; kb < kb1 && ok; ++kb) {
            ok = put_stage(jb, p.prog.pa[step], p.prog.pb[step], kt);
            if (++kt == KTS) {
              kt = 0;
              ++step;
            }
          }
        }
      }
      if (!ok && leader) {
        // let copies already issued land before shared memory is released (the
        // leader's full barriers count both CTAs' copies)
        for (int st = 0; st < Cfg::STAGES; ++st) {
          if (armed & (1u << st)) {
            const uint32_t par = (armed_par >> st) & 1u;
            const uint64_t dl = globaltimer() + 100000000ull;
            while (!mbar_try_wait(full_bar(st), par) && globaltimer() < dl) {
            }
          }
        }
      }
      if (PAIR && ok) {
        // the leader's commits arrive on this CTA's empty barriers: wait until
        // every stage is released, so no arrival is left in flight at exit
        for (int i = 0; i < Cfg::STAGES && ok; ++i) {
          ok = wait_bar<PAIR>(empty_bar(stage), phase ^ 1u, abort_flag, p);
          if (++stage == Cfg::STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // The whole warp walks the loops and an elected lane issues: descriptors and
    // barrier addresses are then the same for all lanes, and the compiler keeps
    // them in the uniform registers that the tensor instructions take.
    if (leader) {
      constexpr uint32_t idesc = F8 ? idesc_e4m3(Cfg::BM, BN) : idesc_bf16(Cfg::BM, BN);
      int stage = 0;
      uint32_t phase = 0;
      int buf = 0;
      uint32_t aph0 = 0, aph1 = 0;  // phases of the two accumulators
      bool ok = true;
      bool issued = false;
      auto wait_all = [&](uint32_t bar, uint32_t parity) __attribute__((always_inline)) -> bool {
        return __all_sync(0xffffffffu, wait_bar<PAIR>(bar, parity, abort_flag, p)) != 0;
      };
      // one stage of MMAs; `first` starts a chunk (waits for a free TMEM buffer
      // and overwrites it), `last` ends it (publishes the buffer)
      auto mma_stage = [&](bool first, bool last) __attribute__((always_inline)) -> bool {
        if (first) {
          if (!wait_all(accempty_bar(buf), (buf ? aph1 : aph0) ^ 1u)) return false;
        }
        if (!wait_all(full_bar(stage), phase)) return false;
        tc_fence_after();
        if (elect_one()) {
          const uint32_t sa = sbase + stage * Cfg::STAGE_BYTES;
          const uint32_t d = tmem + static_cast<uint32_t>(buf * BN);
          const uint64_t ad = sdesc_sw128(sa);
          const uint64_t bd = sdesc_sw128(sa + Cfg::A_BYTES);
#pragma unroll
          for (int ks = 0; ks < TC_MMA_PER_ATOM; ++ks) {
            // advance 32 bytes (16 bf16 or 32 e4m3) along K inside the swizzled row
            const uint32_t acc = (first && ks == 0) ? 0u : 1u;
            if (F8) {
              if (PAIR) {
                umma_e4m3_pair(d, ad + 2ull * ks, bd + 2ull * ks, idesc, acc);
              } else {
                umma_e4m3(d, ad + 2ull * ks, bd + 2ull * ks, idesc, acc);
              }
            } else if (PAIR) {
              umma_bf16_pair(d, ad + 2ull * ks, bd + 2ull * ks, idesc, acc);
            } else {
              umma_bf16(d, ad + 2ull * ks, bd + 2ull * ks, idesc, acc);
            }
          }
          if (PAIR) {
            umma_commit_pair_both(empty_bar(stage));
          } else {
            umma_commit(empty_bar(stage));
          }
          if (last) {
            if (PAIR) {
              umma_commit_pair_both(accfull_bar(buf));
            } else {
              umma_commit(accfull_bar(buf));
            }
          }
        }
        __syncwarp();
        issued = true;
        if (last) {
          if (buf) {
            aph1 ^= 1u;
          } else {
            aph0 ^= 1u;
          }
          buf ^= 1;
        }
        if (++stage == Cfg::STAGES) {
          stage = 0;
          phase ^= 1u;
        }
        return true;
      };
      int rslot = 0;
      uint32_t rph = 0;
      for (int it = 0; ok; ++it) {
        int tile = 0, u0 = 0, u1 = 0x7fffffff;
        if constexpr (WALK == 2) {
          if (!wait_all(ring_full(rslot), rph)) {
            ok = false;
            break;
          }
          tile = ring_tile[rslot];
          __syncwarp();
          if (lane == 0) mbar_arrive(ring_empty(rslot));
          if (++rslot == kTileRing) {
            rslot = 0;
            rph ^= 1u;
          }
          if (tile < 0) break;
        } else {
          if (!static_item(it, tile, u0, u1)) break;
        }
        int KT = p.KT;
        if (p.mats != nullptr) {
          const Job jb = job_of<BN, PAIR>(p, &tmA, &tmB, tile, rank);
          if (jb.skip) continue;
          KT = jb.KT;
        }
        const int KTS = KT;  // stages per step
        int base = 0;
        for (int g = 0; g < p.prog.nsegs && ok; ++g) {
          const int nkb = p.prog.seg[g].nsteps * KTS;
          const int nch = (nkb + CHS - 1) / CHS;
          const int lo = max(u0 - base, 0), hi = min(u1 - base, nch);
          base += nch;
          if (lo >= hi) continue;
          const int kb1 = min(hi * CHS, nkb);
          int kc = 0;
          for (int kb = lo * CHS; kb < kb1 && ok; ++kb) {
            ok = mma_stage(kc == 0, kc == CHS - 1 || kb == kb1 - 1);
            if (++kc == CHS) kc = 0;
          }
        }
      }
      if (!ok && issued && elect_one()) {
        // wait for the MMAs in flight before TMEM is released
        if (PAIR) {
          umma_commit_pair_self(drain_bar);
        } else {
          umma_commit(drain_bar);
        }
        const uint64_t dl = globaltimer() + 100000000ull;
        while (!mbar_try_wait(drain_bar, 0) && globaltimer() < dl) {
        }
      }
      if (PAIR && ok) {
        // both epilogues arrive on this CTA's accumulator barriers: wait for
        // their last releases, so no arrival is left in flight at exit
        ok = wait_all(accempty_bar(0), aph0 ^ 1u) && wait_all(accempty_bar(1), aph1 ^ 1u);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    constexpr int COLS = Cfg::COLS;
    const int e = warp - 2;
    const int q = warp & 3;   // TMEM lane quadrant this warp may access
    const int h = e >> 2;     // which half of the BN columns
    const int cbase = h * COLS;
    const uint32_t taddr_row = tmem + (static_cast<uint32_t>(32 * q) << 16);

    int32_t S[COLS];
    int buf = 0;
    uint32_t aph[2] = {0u, 0u};
    bool ok = true;
    // PAIR: TMEM buffers are released on the leader's barrier
    const uint32_t accempty_target0 = PAIR ? map_to_cta(accempty_bar(0), 0) : accempty_bar(0);

    // one finished chunk from TMEM added into the segment's sum S
    auto drain_chunk = [&]() __attribute__((always_inline)) -> bool {
      // one lane polls the barrier (32 pollers per warp would crowd the
      // barrier word the MMA issuer and the copies also use); the warp then
      // synchronises and orders its TMEM loads after that wait (tcgen05.ld
      // below is warp-collective, so the whole warp takes the same branch)
      int got = 0;
      if (lane == 0) got = wait_bar<PAIR>(accfull_bar(buf), aph[buf], abort_flag, p) ? 1 : 0;
      got = __shfl_sync(0xffffffffu, got, 0);
      if (!got) return false;
      tc_fence_after();
#pragma unroll
      for (int g = 0; g < COLS / 16; ++g) {
        uint32_t v[16];
        tmem_ld16(taddr_row + static_cast<uint32_t>(buf * BN + cbase + 16 * g), v);
        tmem_wait_ld();
#pragma unroll
        for (int t = 0; t < 16; ++t) S[16 * g + t] += __float2int_rn(__uint_as_float(v[t]));
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (PAIR) {
          mbar_arrive_cluster(accempty_target0 + 8u * buf);
        } else {
          mbar_arrive(accempty_bar(buf));
        }
      }
      aph[buf] ^= 1u;
      buf ^= 1;
      return true;
    };

#pragma unroll
    for (int c = 0; c < COLS; ++c) S[c] = 0;
    const uint64_t pol = policy_evict_last();
    int rslot = 0;
    uint32_t rph = 0;
    for (int it = 0; ok; ++it) {
      int tile = 0, u0 = 0, u1 = 0x7fffffff;
      if constexpr (WALK == 2) {
        int got = 0, t = 0;
        if (lane == 0) {
          got = wait_bar<false>(ring_full(rslot), rph, abort_flag, p) ? 1 : 0;
          if (got) {
            t = ring_tile[rslot];
            mbar_arrive(ring_empty(rslot));
          }
        }
        got = __shfl_sync(0xffffffffu, got, 0);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (++rslot == kTileRing) {
          rslot = 0;
          rph ^= 1u;
        }
        if (!got) {
          ok = false;
          break;
        }
        if (t < 0) break;
        tile = t;
      } else {
        if (!static_item(it, tile, u0, u1)) break;
      }
      int KT = p.KT;
      if (p.mats != nullptr) {
        const Job jb = job_of<BN, PAIR>(p, &tmA, &tmB, tile, rank);
        if (jb.skip) continue;
        KT = jb.KT;
      }
      const int KTS = KT;
      // the group sums of this CTA's part of the tile; element c of this thread
      // at [32 c] (a warp touches 256 contiguous bytes per column)
      long long* part = p.area + (static_cast<int64_t>(tile) * Cfg::RANKS + rank) * p.prog.ng * Cfg::PART +
                        e * (COLS * 32) + lane;
      int base = 0;
      for (int g = 0; g < p.prog.nsegs && ok; ++g) {
        const TcSeg& seg = p.prog.seg[g];
        const int nch = (seg.nsteps * KTS + CHS - 1) / CHS;
        const int lo = max(u0 - base, 0), hi = min(u1 - base, nch);
        base += nch;
        if (lo >= hi) continue;
        for (int ch = lo; ch < hi && ok; ++ch) ok = drain_chunk();
        if (!ok) break;
        // ---- add the exact sum to the tile's groups at L2 (red: nothing comes
        // back, so the adds cost no round trip)
        for (int i = 0; i < 3; ++i) {
          const long long w = seg.w[i];
          if (w == 0) continue;
          long long* area = part + (seg.g0 + i) * Cfg::PART;
#pragma unroll
          for (int c = 0; c < COLS; ++c) red_add_keep(area + 32 * c, static_cast<long long>(S[c]) * w, pol);
        }
#pragma unroll
        for (int c = 0; c < COLS; ++c) S[c] = 0;
      }
    }
  }

  // ------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();  // neither CTA leaves while the other may still use its barriers or TMEM
  if (warp == 1) {
    tc_fence_after();
    if (PAIR) {
      tmem_dealloc_pair(tmem, Cfg::TMEM_COLS);
    } else {
      tmem_dealloc(tmem, Cfg::TMEM_COLS);
    }
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (fn == nullptr) {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  }
  return fn;
}

// 2-D view of s stacked digit planes (bf16, or E4M3 bytes when f8): dim0 = k_pad
// (contiguous), dim1 = s * rows; boxes of one 128-byte row by box_rows.
bool make_plane_map(CUtensorMap* tm, const void* planes, int64_t k_pad, int64_t rows_total, int box_rows,
                    bool f8 = false) {
  auto fn = encode_fn();
  if (fn == nullptr) return false;
  const int eb = f8 ? 1 : 2;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(k_pad), static_cast<cuuint64_t>(rows_total)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(k_pad * eb)};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(TC_ROW_BYTES / eb), static_cast<cuuint32_t>(box_rows)};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(tm, f8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                  const_cast<void*>(planes), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace

bool make_plane_map_ext(CUtensorMap* tm, const void* planes, int64_t k_pad, int64_t rows_total, int box_rows,
                        bool f8) {
  return make_plane_map(tm, planes, k_pad, rows_total, box_rows, f8);
}

namespace {
// Exact bound of a product's combined integer sum_L S_L 2^(beta (s+1-L)): whether
// it fits a signed 64-bit word (then one group sum per element is enough).
bool one_word(int s, int beta, int64_t k) {
  const double dmax = beta == 7 ? 127.0 : (beta == 8 ? 128.0 : 16.0);
  double t = 0.0;
  for (int L = 2; L <= s + 1; ++L) t += (L - 1) * std::ldexp(1.0, beta * (s + 1 - L));
  return t * dmax * dmax * static_cast<double>(k) < 9.0e18;
}

// Levels s+1 .. 2, one segment each: the pairs (i, j) with i + j = L.
void direct_program(int s, int beta, int group, int64_t k, bool levels, TcProgram& pr) {
  std::memset(&pr, 0, sizeof(pr));
  const int groups = (s + group - 1) / group;
  const bool one = groups <= 2 && one_word(s, beta, k);
  pr.ng = levels ? s : (one ? 1 : groups);
  int step = 0;
  for (int L = s + 1; L >= 2; --L) {
    TcSeg& g = pr.seg[pr.nsegs++];
    const int pos = s + 1 - L;
    g.step0 = step;
    for (int i = std::max(1, L - s); i <= std::min(s, L - 1); ++i) {
      pr.pa[step] = static_cast<unsigned char>(i - 1);
      pr.pb[step] = static_cast<unsigned char>(L - i - 1);
      ++step;
    }
    g.nsteps = step - g.step0;
    g.g0 = levels ? L - 2 : (one ? 0 : pos / group);
    g.w[0] = levels ? 1 : 1ll << (beta * (one ? pos : pos % group));
  }
}

// The same sums with difference products (see diff_planes): the digit products
// A_i B_i with the weights of every level they enter, the differences of each
// level with its negative weight, and the pairs (1, s), (s, 1) as they are.
// Twice the adds of the direct program (2 s - 1 segments instead of s) for a
// quarter to a third fewer products.
void diff_program(int s, int beta, int group, int64_t k, TcProgram& pr) {
  std::memset(&pr, 0, sizeof(pr));
  const int groups = (s + group - 1) / group;
  const bool one = groups <= 2 && one_word(s, beta, k);
  pr.ng = one ? 1 : groups;
  int step = 0;
  auto add_step = [&](int a, int b) {
    pr.pa[step] = static_cast<unsigned char>(a);
    pr.pb[step] = static_cast<unsigned char>(b);
    ++step;
  };
  auto open = [&]() -> TcSeg& {
    TcSeg& g = pr.seg[pr.nsegs++];
    g.step0 = step;
    return g;
  };
  auto weigh = [&](TcSeg& g, int L, int sign) {
    const int pos = s + 1 - L;
    g.w[one ? 0 : pos / group] += sign * (1ll << (beta * (one ? pos : pos % group)));
  };
  for (int i = 1; i < s; ++i) {
    TcSeg& g = open();
    add_step(i - 1, i - 1);
    g.nsteps = 1;
    for (int j = 1; j < s && i + j <= s + 1; ++j) weigh(g, i + j, 1);
  }
  {
    TcSeg& g = open();
    add_step(0, s - 1);
    add_step(s - 1, 0);
    g.nsteps = 2;
    weigh(g, s + 1, 1);
  }
  for (int L = s + 1; L >= 3; --L) {
    TcSeg& g = open();
    for (int i = 1; 2 * i < L; ++i) {
      const int j = L - i;
      if (j < s) add_step(diff_plane(s, i, j), diff_plane(s, i, j));
    }
    g.nsteps = step - g.step0;
    weigh(g, L, -1);
  }
}

int chunk_atoms(int beta) { return beta == 5 ? 64 : 16; }

void group_scales(TcParams& p) {
  for (int g = 0; g < 3; ++g) p.gscale[g] = std::ldexp(1.0, -p.beta * (p.s + 1 - p.group * g));
}

// fp32 chunks of one tile (split launches)
int chunk_count(const TcProgram& pr, int kts, int chs) {
  int cnt = 0;
  for (int g = 0; g < pr.nsegs; ++g) cnt += (pr.seg[g].nsteps * kts + chs - 1) / chs;
  return cnt;
}

// Set before every launch rather than once per process: the attribute belongs
// to the kernel as loaded in the current context, and a context created anew
// (after cudaDeviceReset) starts from the default limit. The call is host-side
// only and costs about a microsecond against milliseconds of kernel.
template <int BN, bool PAIR, bool F8 = false, int WALK = 0>
cudaError_t set_smem_attr() {
  return cudaFuncSetAttribute(ozaki_tc_kernel<BN, PAIR, F8, WALK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              TcCfg<BN, PAIR, F8>::SMEM);
}

// The launch configuration of the product kernel (clusters of two CTAs for PAIR).
template <int BN, bool PAIR, bool F8>
struct TcLaunch {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[2];
  TcLaunch(int grid, cudaStream_t st, bool chained = false) {
    std::memset(&cfg, 0, sizeof(cfg));
    std::memset(at, 0, sizeof(at));
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(TC_THREADS);
    cfg.dynamicSmemBytes = TcCfg<BN, PAIR, F8>::SMEM;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = PAIR ? 2 : 1;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = chained ? 2 : 1;
  }
};

template <int BN, bool PAIR, int OUT>
void launch_finish(const TcParams& p, cudaStream_t st) {
  const int grid = p.ntiles * (TcCfg<BN, PAIR>::BM / 32) * (BN / 32);
  auto launch = [&](void (*kernel)(TcParams)) {
    if (p.mats == nullptr) {
      launch_chained(kernel, grid, FIN_THREADS, st, p);
    } else {
      kernel<<<grid, FIN_THREADS, 0, st>>>(p);
    }
  };
  if (OUT == OUT_STORE && p.mats == nullptr && p.epi.kind == EPI_LEVELS) {
    launch(ozaki_finish_kernel<BN, PAIR, OUT_STORE, 0>);
  } else if (p.prog.ng == 1) {
    launch(ozaki_finish_kernel<BN, PAIR, OUT, 1>);
  } else if (p.prog.ng == 2) {
    launch(ozaki_finish_kernel<BN, PAIR, OUT, 2>);
  } else {
    launch(ozaki_finish_kernel<BN, PAIR, OUT, 3>);
  }
}

// The product kernel on `grid` CTAs, then the finish kernel over its tiles.
template <int BN, bool PAIR = false, bool F8 = false, int WALK = 0>
cudaError_t launch_tc_impl(const CUtensorMap& ta, const CUtensorMap& tb, const TcParams& p, int grid, cudaStream_t st) {
  cudaError_t e = set_smem_attr<BN, PAIR, F8, WALK>();
  if (e != cudaSuccess) return e;
  TcLaunch<BN, PAIR, F8> l(grid, st, p.mats == nullptr);  // (a batch's products are captured in a graph's loop)
  e = cudaLaunchKernelEx(&l.cfg, ozaki_tc_kernel<BN, PAIR, F8, WALK>, ta, tb, p);
  if (e != cudaSuccess) return e;
  const int kind = p.mats != nullptr ? (p.phase != 0 ? EPI_PM_UPDATE : EPI_SYM_STORE) : p.epi.kind;
  if (kind == EPI_PM_UPDATE) {
    launch_finish<BN, PAIR, OUT_UPDATE>(p, st);
  } else if (kind == EPI_CHEB) {
    launch_finish<BN, PAIR, OUT_CHEB>(p, st);
  } else {
    launch_finish<BN, PAIR, OUT_STORE>(p, st);
  }
  count_launch(2);
  return cudaGetLastError();
}

bool g_pairing = true;

// One-shot stall test (dmp_test_stall_next_product): wait limit in microseconds
// for the next tcgen05 product launch, 0 = off.
std::atomic<int> g_stall_us{0};

// CTA pairs of the pair kernel that can be resident at once (0: none)
int tc_max_pairs() {
  static const int pairs = [] {
    int found = 0;
    if (set_smem_attr<256, true>() == cudaSuccess) {
      TcLaunch<256, true, false> l(2, nullptr);
      int c = 0;
      if (cudaOccupancyMaxActiveClusters(&c, ozaki_tc_kernel<256, true>, &l.cfg) == cudaSuccess) found = c;
    }
    (void)cudaGetLastError();
    return std::min(found, kTcMaxCtas / 2);
  }();
  return pairs;
}

}  // namespace

bool tc_pairs_available() { return g_pairing && tc_max_pairs() > 0; }

int set_stall_test(int wait_limit_us) {
  if (wait_limit_us < 0) return DMP_ERR_INVALID_ARG;
  g_stall_us.store(wait_limit_us);
  return DMP_OK;
}

int set_tc_pairing(int enable) {
  const int prev = g_pairing ? 1 : 0;
  g_pairing = enable != 0;
  return prev;
}

int tc_max_ctas() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  return std::min(sms, kTcMaxCtas);
}

// 80 MiB: 160 pair tiles of one group sum per element, two waves of the pair
// kernel, which stay in the 129 MB L2 between the product and its output step, or
// 80 of two. With three that is 53 tiles: 23 of the 76 pairs of every launch have
// none of their own, and a batch's tiles are walked whole. 120 MiB hold a whole
// wave. Batch of two matrices of n = 4096 (272 tiles, 8 iterations), 80 against 120
// MiB: 9 and 11 E4M3 slices 57.9 / 45.3 and 77.5 / 59.7 ms, 9 INT8 slices 97.2 /
// 72.6. (For single matrices see wants_wave in api.cu.)
size_t tc_area_bytes(bool wave) {
  return static_cast<size_t>(kTcMaxCtas) * (wave ? 3 : 2) * TC_BM * 256 * sizeof(long long);
}
bool tc_wants_wave(int s, int beta, int64_t tiles) {
  return s > 2 * (beta == 8 ? 3 : 4) && tiles * 3 * (2 * TC_BM) * 256 * sizeof(long long) > tc_area_bytes(false);
}

bool g_split_tiles = true;

int set_tc_split_tiles(int enable) {
  const int prev = g_split_tiles ? 1 : 0;
  g_split_tiles = enable != 0;
  return prev;
}

// The group sums of the next `bytes` of the area are zero before a launch adds
// to them: cleared here once per call, by the finish kernel after that.
cudaError_t tc_area_clear(TcArea& a, size_t bytes, cudaStream_t st) {
  if (bytes <= a.clean) return cudaSuccess;
  const size_t front = a.clean == 0 ? a.front : 0;
  const cudaError_t e = cudaMemsetAsync(static_cast<char*>(a.ptr) + a.clean - front, 0, bytes - a.clean + front, st);
  if (e == cudaSuccess) a.clean = bytes;
  return e;
}

namespace {

// Length of the equal parts of a split tile's `units` (TcParams::head_len): the
// one for which the longest share is shortest, the rest of the nsplit tiles
// going to `extra` CTAs (none: the parts cover the tile).
int head_length(int units, int nsplit, int heads, int extra) {
  const int most = (units + heads - 1) / heads;
  if (extra <= 0) return most;
  int best = most, best_share = most;
  for (int h = 1; h < most; ++h) {
    const int64_t rest = static_cast<int64_t>(nsplit) * (units - heads * h);
    const int share = std::max(h, static_cast<int>((rest + extra - 1) / extra));
    if (share < best_share) {
      best = h;
      best_share = share;
    }
  }
  return best;
}

// The part of the area that a launch fills: with one or two group sums the 80 MiB
// that stay in L2.
size_t area_room(const TcArea& a, int ng) { return ng > 2 ? a.bytes : std::min(a.bytes, tc_area_bytes(false)); }

// Operand planes up to this size stay in L2 while a product runs.
constexpr double kL2Planes = 70e6;

// One single-matrix product on tiles of BM x BN.
template <int BN, bool PAIR, bool F8>
cudaError_t run_product(const void* A, const void* B, int64_t k_pad, int planes, TcParams& p,
                        TcArea& area, cudaStream_t st) {
  using Cfg = TcCfg<BN, PAIR, F8>;
  CUtensorMap ta, tb;
  if (!make_plane_map(&ta, A, k_pad, planes * p.rows_a, TC_BM, F8)) return cudaErrorInvalidValue;
  if (!make_plane_map(&tb, B, k_pad, planes * p.rows_b, PAIR ? BN / 2 : BN, F8)) return cudaErrorInvalidValue;
  const int units = PAIR ? tc_max_pairs() : tc_max_ctas();
  TileOrder order(p.m, p.n, Cfg::BM, BN, p.sym != 0, units);
  const int64_t ntiles = order.count();
  p.column_bits = order.column_bits();
  if (p.column_bits < 0) return cudaErrorInvalidValue;
  // While there are fewer tiles than CTAs, chunks no longer than a CTA's share of
  // the K atoms (half of it on 256-column tiles, where an added chunk costs less
  // than an uneven share: n = 1024, E4M3, s = 9 62 -> 58 us).
  if (g_split_tiles && ntiles < units) {
    int steps = 0;
    for (int g = 0; g < p.prog.nsegs; ++g) steps += p.prog.seg[g].nsteps;
    const int64_t atoms = static_cast<int64_t>(steps) * p.KT * ntiles;
    const int cut = (BN < 256 ? 1 : 2) * units;
    p.CH = static_cast<int>(std::min<int64_t>(p.CH, std::max<int64_t>(BN < 256 ? 1 : 2, (atoms + cut - 1) / cut)));
  }
  p.units = chunk_count(p.prog, p.KT, p.CH);
  const double plane_bytes = static_cast<double>(k_pad) * (F8 ? 1 : 2) * planes * (p.m + (A == B ? 0 : p.n));

  // rounds of as many tiles as the area holds group sums for, in whole waves
  const size_t tile_bytes = static_cast<size_t>(Cfg::RANKS) * p.prog.ng * Cfg::PART * sizeof(long long);
  int per = static_cast<int>(
      std::min<int64_t>(std::min<int64_t>(ntiles, kMaxLaunchTiles), area_room(area, p.prog.ng) / tile_bytes));
  if (per <= 0) return cudaErrorInvalidValue;
  if (per < ntiles && per > units) per = per / units * units;
  cudaError_t e = tc_area_clear(area, per * tile_bytes, st);
  for (int64_t t0 = 0; t0 < ntiles && e == cudaSuccess; t0 += per) {
    p.ntiles = static_cast<int>(std::min<int64_t>(per, ntiles - t0));
    for (int t = 0; t < p.ntiles; ++t) p.at[t] = pack_tile(order.next(), p.column_bits);
    p.nwhole = g_split_tiles ? p.ntiles / units * units : p.ntiles;
    const int nsplit = p.ntiles - p.nwhole;
    // The tiles of a partial wave are shared by all CTAs. While the planes stay
    // in L2, all their units are one sequence, evenly cut (n = 1792: 98 us per
    // product against 105 for two CTAs per tile). Otherwise a CTA takes the same
    // part of its tile as the others, so that they walk the same planes at the
    // same K and share their panels (out of step they stream them from HBM: n =
    // 4096 754 us against 633 for one CTA per tile), and what that leaves of
    // each tile goes to the CTAs that are left.
    p.heads = p.head_len = 0;
    const int64_t split_units = static_cast<int64_t>(nsplit) * p.units;
    if (nsplit > 0 && plane_bytes > kL2Planes) {
      p.heads = std::min(p.units, units / nsplit);
      p.head_len = head_length(p.units, nsplit, p.heads, units - nsplit * p.heads);
    }
    int grid = units;
    if (p.nwhole == 0) {
      grid = static_cast<int>(std::min<int64_t>(units, split_units));
    } else if (!g_split_tiles) {
      grid = std::min(units, p.nwhole);
    }
    e = launch_tc_impl<BN, PAIR, F8>(ta, tb, p, (PAIR ? 2 : 1) * grid, st);
  }
  return e;
}

}  // namespace

cudaError_t launch_ozaki_tc(const void* A, const void* B, const int32_t* ea, const int32_t* eb, int64_t m,
                            int64_t n, int64_t k, int64_t rows_a, int64_t rows_b, int64_t k_pad, int s, int beta,
                            bool diff, int sym, const EpiArgs& epi, const int* done, int* err, TcArea& area,
                            cudaStream_t st) {
  if (m <= 0 || n <= 0) return cudaSuccess;
  const bool f8 = beta == 5;  // E4M3 nearest digits
  const int atom_k = f8 ? 128 : TC_BK;
  if (rows_a % TC_BM != 0 || rows_b % 256 != 0 || k_pad % atom_k != 0) return cudaErrorInvalidValue;
  // products run on CTA pairs (256 x 256 tiles, 2-SM MMA) when rows allow
  const bool pair = g_pairing && rows_a % (2 * TC_BM) == 0 && k_pad % (2 * atom_k) == 0 && tc_max_pairs() > 0;
  TcParams p;
  std::memset(&p, 0, sizeof(p));
  p.s = s;
  p.beta = beta;
  p.KT = static_cast<int>(k_pad / atom_k);
  // K chunk in atoms: 1024 (beta 7: 127^2; beta 8 nearest: 128^2) K elements, of
  // up to 65536 (beta 5 nearest: 16^2) 8192 so that tiles can be shared in fine
  // parts, keep every fp32 partial sum at most 2^24
  p.CH = chunk_atoms(beta);
  p.group = beta == 8 ? 3 : 4;
  group_scales(p);
  p.m = m;
  p.n = n;
  p.rows_a = rows_a;
  p.rows_b = rows_b;
  p.sym = sym;
  p.ea = ea;
  p.eb = eb;
  p.epi = epi;
  p.done = done;
  p.err = err;
  p.area = static_cast<long long*>(area.ptr);
  p.timeout_ns = 5000000000ull;
  // the stall test is taken by a launch that runs now, never by one being
  // captured into a graph (every replay would stall)
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
    if (const int us = g_stall_us.exchange(0); us > 0) {
      p.stall_test = 1;
      p.timeout_ns = 1000ull * static_cast<unsigned long long>(us);
    }
  }
  // the test hook for the level sums takes the pairs one by one
  diff = diff && epi.kind != EPI_LEVELS;
  if (diff) {
    diff_program(s, beta, p.group, k, p.prog);
  } else {
    direct_program(s, beta, p.group, k, epi.kind == EPI_LEVELS, p.prog);
  }
  const int planes = s + (diff ? diff_planes(s) : 0);
  ProfScope prof(DMP_PROF_PRODUCT, st);
  // Few tiles: smaller ones, whose group sums a CTA adds in proportion faster
  // (a 128 x 256 part takes it 6 us, 128 x 64 1.5 us) and whose operands more CTAs
  // share; larger outputs want the pair kernel's fewer bytes per product. Per
  // product, INT8 s = 5, pair / 128 x 128 / 128 x 64 tiles: n = 256 22.9 / 18.1 /
  // 16.1 us, n = 384 25.1 / 19.5 / 19.0, n = 512 27.7 / 21.5 / 25.5, n = 768 34.5 /
  // 30.4 / 34.4, n = 1024 41.0 / 42.7 / 52.2; the other modes alike.
  // With a short K the adds outweigh the products on larger outputs as well, as
  // long as the 128 x 128 tiles are one wave. 128 x 128 against pair tiles, us: 1000
  // x 333 x 257 BF16 s = 6 31.6 / 43.6, 2000 x 700 x 128 INT8 s = 7 48 / 58, 1000 x
  // 500 x 257 E4M3 s = 8 35.6 / 44; level at 1000 x 1000 x 257 INT8 52 / 50, behind
  // at 900 x 900 x 300 E4M3 54 / 46 and 2500 x 1000 x 96 INT8 (160 tiles) 61 / 58.
  const int64_t tm = (m + 255) / 256, tn = (n + 255) / 256;
  const int64_t big_tiles = sym ? tn * (tn + 1) / 2 : tm * tn;
  if (pair && big_tiles <= 1)
    return f8 ? run_product<64, false, true>(A, B, k_pad, planes, p, area, st)
              : run_product<64, false, false>(A, B, k_pad, planes, p, area, st);
  const bool short_k = !sym && big_tiles * k <= 4096 && ((m + 127) / 128) * ((n + 127) / 128) <= tc_max_ctas();
  if (pair && (big_tiles <= 6 || short_k))
    return f8 ? run_product<128, false, true>(A, B, k_pad, planes, p, area, st)
              : run_product<128, false, false>(A, B, k_pad, planes, p, area, st);
  if (pair)
    return f8 ? run_product<256, true, true>(A, B, k_pad, planes, p, area, st)
              : run_product<256, true, false>(A, B, k_pad, planes, p, area, st);
  return f8 ? run_product<256, false, true>(A, B, k_pad, planes, p, area, st)
            : run_product<256, false, false>(A, B, k_pad, planes, p, area, st);
}

cudaError_t launch_ozaki_tc_grouped(const BatchMat* mats, const int4* tiles, int ntiles, int64_t nmax, int bn,
                                    bool pair, int beta, int s, int phase, int cur, int* err, TcArea& area,
                                    int* counter, cudaStream_t st) {
  if (ntiles <= 0) return cudaSuccess;
  if (pair && (bn != 256 || tc_max_pairs() <= 0)) return cudaErrorInvalidValue;
  if (beta == 5 && bn != 256) return cudaErrorInvalidValue;  // E4M3 digits: 256-column tiles
  TcParams p;
  std::memset(&p, 0, sizeof(p));
  p.s = s;
  p.beta = beta;
  p.CH = chunk_atoms(beta);
  p.group = beta == 8 ? 3 : 4;
  group_scales(p);
  p.sym = 1;
  p.units = 1;
  p.mats = mats;
  p.tiles = tiles;
  p.phase = phase;
  p.cur = cur;
  p.err = err;
  p.area = static_cast<long long*>(area.ptr);
  p.timeout_ns = 5000000000ull;
  p.tile_counter = counter;
  direct_program(s, beta, p.group, nmax, false, p.prog);
  CUtensorMap unused;
  std::memset(&unused, 0, sizeof(unused));
  const int units = pair ? tc_max_pairs() : tc_max_ctas();
  const size_t tile_bytes = static_cast<size_t>(pair ? 2 : 1) * p.prog.ng * TC_BM * bn * sizeof(long long);
  int per = static_cast<int>(std::min<size_t>(ntiles, area_room(area, p.prog.ng) / tile_bytes));
  if (per <= 0) return cudaErrorInvalidValue;
  if (pair && per < ntiles && per > units) per = per / units * units;
  ProfScope prof(DMP_PROF_PRODUCT, st);
  cudaError_t e = tc_area_clear(area, per * tile_bytes, st);
  for (int t0 = 0; t0 < ntiles && e == cudaSuccess; t0 += per) {
    p.tile0 = t0;
    p.ntiles = p.nwhole = std::min(per, ntiles - t0);
    const int grid = std::min(p.ntiles, units);
    if (pair) {
      // CTA pairs (256-row tiles, 256 columns): the pairs walk the list (largest
      // matrices first) round robin
      e = beta == 5 ? launch_tc_impl<256, true, true>(unused, unused, p, 2 * grid, st)
                    : launch_tc_impl<256, true, false>(unused, unused, p, 2 * grid, st);
      continue;
    }
    // single CTAs take tiles from a counter as they free up (the tiles differ in
    // work: the list holds the largest matrices' tiles first)
    e = cudaMemsetAsync(counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    if (beta == 5) {
      e = launch_tc_impl<256, false, true, 2>(unused, unused, p, grid, st);
    } else if (bn == 128) {
      e = launch_tc_impl<128, false, false, 2>(unused, unused, p, grid, st);
    } else {
      e = launch_tc_impl<256, false, false, 2>(unused, unused, p, grid, st);
    }
  }
  return e;
}

}  // namespace dmp
