// Tensor-core kernels of the FAAR layer step for sm_100a.
//
// One persistent, warp-specialised kernel computes C[M,N] = A[M,Kc] * B[N,Kc]^T for BF16 operands that
// both have the contraction dimension contiguous.  It runs as clusters of two CTAs that share one
// 256 x bn output tile (tcgen05 cta_group::2): CTA r of the pair loads rows [128 r, 128 r + 128) of the
// A tile and rows [bn/2 r, bn/2 (r+1)) of the B tile into its own shared memory, the leader CTA (r = 0)
// issues the 256 x bn x 16 MMAs for both, and each CTA ends up with its 128 accumulator rows x bn
// columns (FP32) in its own tensor memory.  Halving the B tile per CTA halves the shared-memory
// traffic per flop, which is what bounds a single-CTA 128 x 256 tile.
//   warp 0      : TMA producer  (cp.async.bulk.tensor, 128-byte swizzle, multi-stage ring; both CTAs,
//                                both crediting the leader's "full" barrier)
//   warp 1      : MMA issuer    (leader CTA only; tcgen05.mma kind::f16, tcgen05.commit to the
//                                "empty" / "accumulator full" barriers of both CTAs)
//   warps 2..   : epilogue      (tcgen05.ld; two accumulator buffers, so the epilogue of one tile
//                                overlaps the main loop of the next)
// A REF or BWD launch with few tiles and a long contraction splits it (p.splits = 2 or 4): the pairs of a cluster of 4 or 8 CTAs take
// a part of the k blocks of the SAME tile each, then every CTA sends the accumulator columns that are another pair's
// to finish to that pair's CTA of the same rows (distributed shared memory) and finishes its
// own share of the columns, adding the parts in a fixed order (see exchange_parts).
// The three epilogues are the operations of the layer step:
//   REF : Y_fp = X W^T                                   (Procedure step 8)
//   FWD : r = Y_q - Y_ref, sum r^2, dY = 2c r -> dY^T     (steps 9-10, Eq. 5 first term)
//   BWD : G = dY^T X -> dV -> optimiser update + clip     (step 13, Eq. 5, with Eq. 2/3 chain rule)
// In FWD and BWD the accumulator row (TMEM lane) is the output feature o.  In REF it is a row of the result as it lies in
// memory (a token, or an output feature if the target is wanted transposed), so that a lane's 16 columns are contiguous, or
// a column of it where rows are few or off 16 bytes (see result_columns).
//
// Every wait on an mbarrier is bounded: after about two seconds the waiting thread records a code in
// the status word, raises a CTA-wide abort flag and every role leaves its loop; both CTAs then meet at
// the closing cluster barrier, free their tensor memory and exit.
#include <cuda.h>

#include "faar_internal.cuh"

namespace {

constexpr int BM = 128;                // accumulator rows per CTA; the CTA pair covers 256
constexpr int BK = 64;                 // 64 bf16 = one 128-byte swizzle row
constexpr int UMMA_K = 16;
constexpr unsigned long long WAIT_LIMIT_NS = 2000000000ull;
constexpr int PW = 64;                         // BWD epilogue: columns of a staged panel of G
constexpr int PANEL_BYTES = 32 * PW * 4;       // one 32-row x PW-column FP32 panel per TMEM lane quarter
constexpr int SMEM_LIMIT = 227 * 1024;
constexpr int CTL_BYTES = 512;
constexpr int MAX_EPI_WARPS = 16;
constexpr int MAX_STAGES = 10;
constexpr int FIN_COUNT_BITS = 9;              // CTAs of a launch: below 512

// The tile width bn (accumulator columns, a multiple of 16 up to 256) is a launch parameter chosen by
// the host (pick_bn).  Shared memory and tensor memory are laid out for the widest tile.
constexpr int BN_MAX = 256;
// WIDE: the pair's tile is 256 x (288 .. 512), the whole of tensor memory as ONE accumulator (column halves of 256 and of
// the rest, at least 32, each fed by its own MMA from the same A stage).  A stage then holds this CTA's rows of both B halves.
// Per flop the tile pulls a quarter less operand data through the SM than a 256 x 256 tile, which is what
// bounds these kernels; the price is that the epilogue of a tile no longer overlaps the next tile's main loop
// (the two halves drain one after the other while the issuer waits).
constexpr int WIDE_BN = 2 * BN_MAX;
constexpr int WIDE_BN_MIN = BN_MAX + 32;       // no other launch gives a pair of CTAs an MMA of fewer than 32 columns either
// The tile forms of a launch, chosen at compile time (as run-time options of one kernel they cost the others time): tiles of
// up to 256 columns, 256 x (288 .. 512), a contraction split over the pairs of a cluster, or (BWD) 256-wide tiles of a short contraction.
//
// SHORT_TILES: a dW launch of few k blocks is bound by its epilogue's state traffic.  What limits that is the L1 cache: a
// load in flight holds its L1 lines, and with all of an SM's 256 KB but 28 taken as shared memory, loads beyond about 24 KB
// wait to be issued (1000 clocks per instruction of 4 weights a lane).  So a short contraction gives up one stage of the ring,
// the next smaller carve-out leaves 60 KB of L1, and a lane requests 8 weights at a time, in 32-byte accesses.
// dW kernel of 8192 x 2048, us: 64 tokens 93.3 -> 75.9 (4.5 -> 5.4 TB/s of state), 1024 95.3 -> 82.1, 2048 100.8 -> 93.8, 3000
// 130.0 -> 128.9, 4096 134 -> 137; of 12288 x 2048 at 2000 149 -> 143.  With the carve-out but 4 weights at a time 64 tokens
// take 91.8, with 8 at a time but no carve-out 97.6; without another stage (92 KB of L1) nothing changes but 2000 tokens, 148.
// Above SHORT_BLOCKS the main loop needs the stage: operands and state together then take all the 64 bytes a clock that an
// SM draws from L2.  The line is the same for plain gradient descent, a third of the state, us: 64 tokens 51.9 -> 38.9, 1024
// 58.2 -> 46.0, 2048 67.9 -> 62.4, 2560 74.9 -> 73.1 (Adam 107.0 -> 104.7, writing the next operand too 116.3 -> 115.4).
//
// SPLIT_NARROW: a split contraction that leaves a CTA at most 32 columns to finish, of a dW launch.  The lanes of its epilogue then
// cover 16 or 32 columns of a row instead of 64, most of which there would be none of: a small layer's epilogue executed the
// instructions of four times its weights.  Step of 128 x 256 at 1024 tokens (16 columns) 14.75 -> 12.6 us; dW kernel (shares of 16
// columns) of 256 x 256 at 1024 tokens 9.7 -> 7.9, 128 x 256 at 4096 12.3 -> 10.7, 256 x 1024 at 1024 10.0 -> 8.9, (of 32) 128 x 1536 at 1536
// 11.1 -> 10.0, 300 x 464 at 2600 12.6 -> 11.6.  (As a choice inside SPLIT_TILES it cost shares of 64 columns 2 %.)
constexpr int PLAIN_TILES = 0, WIDE_TILES = 1, SPLIT_TILES = 2, SHORT_TILES = 3, SPLIT_NARROW = 4;
constexpr int SHORT_BLOCKS = 40;
constexpr int SHORT_SMEM = 387 * 512;          // with the system's 1 KB below the 196 KB carve-out
constexpr int SHORT_CARVEOUT = 85;             // percent of the 228 KB: 193.8, which is rounded up to the size on offer, 196 KB
constexpr int GATED_FWD = 8, GATED_BWD = 10, ROPE = 16, STATS = 32, SUMS = 66;   // MN (see the kernel) of the gated product's launches, of q / k / v's, of
// logits', of the attention output's gradient
constexpr int GATE_COLS = 32, GATE_PANEL = 32 * GATE_COLS * 2;        // backward: a warp's 32 rows x 32 columns in BF16
template <int MODE, int SHAPE = PLAIN_TILES, int MN = 0> struct Cfg {
  static constexpr bool WIDE = SHAPE == WIDE_TILES, SHORT = SHAPE == SHORT_TILES, SPLIT = SHAPE == SPLIT_TILES || SHAPE == SPLIT_NARROW;
  static constexpr int EPI_WARPS = MODE == FAAR_GEMM_BWD || MN == GATED_BWD ? 16 : 8;
  static constexpr int THREADS = 32 * (2 + EPI_WARPS);
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int BH_BYTES = (BN_MAX / 2) * BK * 2;       // this CTA's 128 rows of one 256-column B tile
  static constexpr int B_BYTES = WIDE ? 2 * BH_BYTES : BH_BYTES;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int LANE_WEIGHTS = SHORT ? 8 : 4;             // BWD: weights of one instruction's state per lane
  static constexpr int EPI_BYTES = MODE == FAAR_GEMM_BWD ? 4 * PANEL_BYTES : (MN == GATED_BWD ? EPI_WARPS * GATE_PANEL : 0);
  // The ring: as many stages of the launch's tile width as fit (a stage is the A rows plus bn / 2 rows of B: 32 KB for
  // 256 columns, 18 KB for 32), at most MAX_STAGES.  A small launch's main loop runs at stages / latency, so narrow
  // tiles get the deeper ring.
  static constexpr int RING_BYTES = ((SHORT ? SHORT_SMEM : SMEM_LIMIT) - 1024 - CTL_BYTES - EPI_BYTES) / 1024 * 1024;
  static constexpr int MIN_STAGES = RING_BYTES / STAGE_BYTES;
  static constexpr int TMEM_COLS = 2 * BN_MAX;                 // two accumulator buffers
  static constexpr int COL_GROUPS = EPI_WARPS / 4;             // warps sharing one TMEM lane quarter
  static constexpr int SMEM_BYTES = RING_BYTES + EPI_BYTES + 1024 /*alignment slack*/ + CTL_BYTES;
};

// ---- PTX wrappers ------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address, in CTA `rank` of the cluster, of the object that sits at shared::cta address `addr` here
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
  cluster_arrive_release();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// arrive on a barrier given by its shared::cluster address (this CTA's or the peer's)
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster_addr) : "memory");
}
// the same with what the arriving threads of other CTAs wrote before visible here
__device__ __forceinline__ uint32_t mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return done;
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return done;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

struct AbortCtl {
  volatile int* flag;     // shared memory
  uint32_t* status;       // global status word
  unsigned long long limit_ns = WAIT_LIMIT_NS;
};

// Returns false if the wait was abandoned (time limit, or another thread raised the flag).
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, const AbortCtl& ac, uint32_t code) {
  unsigned long long t0 = global_ns();
  for (uint32_t spin = 1;; ++spin) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((spin & 0xFF) == 0) {
      if (*ac.flag) return false;
      if (global_ns() - t0 > ac.limit_ns) {
        atomicCAS(ac.status, 0u, code);
        *ac.flag = 1;
        return false;
      }
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const AbortCtl& ac, uint32_t code) {
  if (mbar_try_wait(bar, parity)) return true;
  return mbar_wait_slow(bar, parity, ac, code);
}

__device__ __noinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, const AbortCtl& ac, uint32_t code) {
  const unsigned long long t0 = global_ns();
  for (uint32_t spin = 1;; ++spin) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((spin & 0xFF) == 0) {
      if (*ac.flag) return false;
      if (global_ns() - t0 > ac.limit_ns) {
        atomicCAS(ac.status, 0u, code);
        *ac.flag = 1;
        return false;
      }
    }
  }
}
// 16 bytes into another CTA's shared memory, credited there to its barrier `bar`
__device__ __forceinline__ void st_async128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1,%2,%3,%4}, [%5];"
               ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d), "r"(bar) : "memory");
}

// 2-D tiled TMA load into this CTA's shared memory; the byte count is credited to `bar`, which may be
// a barrier of either CTA of the pair (shared::cluster address).  No multicast.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar,
                                            uint64_t l2_policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar), "l"(l2_policy) : "memory");
}
// L2 eviction policies: GEMM operands are re-read by many CTAs and should stay; the per-weight
// optimiser state streams through once per step and should be the first to go.
__device__ __forceinline__ uint64_t l2_policy_keep() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_policy_stream() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
// Four or eight consecutive values of the per-weight state: one access of 16 or 32 bytes, or (`wide` false: a base that is
// off 32 bytes) two of 16.
__device__ __forceinline__ void ldg_state(const float* ptr, bool wide, uint64_t pol, float (&v)[8]) {
  if (wide) {
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], %9;"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "l"(ptr), "l"(pol));
  } else {
#pragma unroll
    for (int h = 0; h < 8; h += 4)
      asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0,%1,%2,%3}, [%4], %5;"
                   : "=f"(v[h]), "=f"(v[h + 1]), "=f"(v[h + 2]), "=f"(v[h + 3]) : "l"(ptr + h), "l"(pol));
  }
}
__device__ __forceinline__ void ldg_state(const float* ptr, bool, uint64_t pol, float (&v)[4]) {
  asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0,%1,%2,%3}, [%4], %5;"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(ptr), "l"(pol));
}
__device__ __forceinline__ void stg_state(float* ptr, bool wide, uint64_t pol, const float (&v)[8]) {
  if (wide) {
    asm volatile("st.global.L2::cache_hint.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8}, %9;" ::"l"(ptr), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "l"(pol) : "memory");
  } else {
#pragma unroll
    for (int h = 0; h < 8; h += 4)
      asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1,%2,%3,%4}, %5;" ::"l"(ptr + h), "f"(v[h]), "f"(v[h + 1]), "f"(v[h + 2]),
                   "f"(v[h + 3]), "l"(pol) : "memory");
  }
}
__device__ __forceinline__ void stg_state(float* ptr, bool, uint64_t pol, const float (&v)[4]) {
  asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1,%2,%3,%4}, %5;" ::"l"(ptr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "l"(pol)
               : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// When all MMAs issued so far have completed, arrive on the barrier at offset `bar` in both CTAs of the pair whose leader
// has cluster rank `leader`.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar, uint32_t leader) {
  const uint16_t mask = (uint16_t)(3u << leader);
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(mask) : "memory");
}
__device__ __forceinline__ void tc_mma_bf16(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate) : "memory");
}
// An instruction of the whole warp.  Rows beyond the matrix take no part in an epilogue's stores, so a __syncwarp stands between
// those and the next load.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ float4 lds128(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

// Shared-memory matrix descriptor: rows of 64 bf16 (128 B) with 128-byte swizzle, contraction
// dimension contiguous; groups of 8 rows are 1024 B apart.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);        // start address
  d |= (uint64_t)1 << 16;                          // leading byte offset (unused with swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;                          // descriptor version for sm_100
  d |= (uint64_t)2 << 61;                          // 128-byte swizzle
  return d;
}
// The same for an operand stored with its M (or N) index contiguous and the contraction index as the row
// ("MN-major"): 64 elements (128 B) of one contraction index form a row, 8 consecutive contraction indices a
// 1024-byte swizzle atom; atoms follow each other along the contraction (stride byte offset, 1024 B: a TMA box
// of 64 x 64 elements lands exactly so) and along M / N (leading byte offset: the next 64-element box, 8192 B on).
__device__ __forceinline__ uint64_t make_smem_desc_mn(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)(8192 >> 4) << 16;                // leading byte offset: next 64 M / N elements
  d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset: next 8 contraction indices
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
constexpr int MN_BOX = 64;                         // M / N elements per MN-major TMA box
constexpr int MN_BOX_BYTES = MN_BOX * BK * 2;      // 8192
__host__ __device__ constexpr int mn_boxes(int columns) { return (columns + MN_BOX - 1) / MN_BOX; }
constexpr uint32_t MN_KSTEP = (UMMA_K * 128) >> 4; // 16 contraction indices on: 2048 B in the address field
// Instruction descriptor: D = F32, A = B = BF16, M = 256 (the CTA pair), N = bn; bits 15 / 16 say that A / B is
// MN-major instead of K-major.
__device__ __forceinline__ uint32_t make_idesc(int bn, int a_mn = 0, int b_mn = 0) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
         ((uint32_t)(bn >> 3) << 17) | ((uint32_t)((2 * BM) >> 4) << 24);
}

// One linear's per-weight state (faar_bwd_state); the bases are moved back by its first row, so that rows of the launch
// index them.
struct Segment {
  float* V; const uint8_t* code; const uint8_t* scales; const float* s_global;
  float* adam_m; float* adam_u; float* dV;
  float lam4;                       // -4 lambda / N: (lambda / N) (4 - 8 v) = lam4 (2 v - 1)
  int wide;                         // V, m, u and dV all lie on 32-byte boundaries (a row is a multiple of 64 bytes)
};

// What a launch needs of the one before it on the stream: everything (0), nothing (BESIDE, see faar_pdl_wait_first), or the A
// operand alone (AHEAD): the first ring of the B operand and what the epilogue asks for ahead (target values, optimiser state) then
// come in under the end of that launch.  Step, us: 128 x 256 at 1024 tokens 12.5 -> 12.0, 512 x 512 at 512 16.1 -> 15.7, 256 x 1024 at 1024
// 16.0 -> 15.6, 64 x 8192 at 300 42.8 -> 41.7, 1000 x 1040 at 777 20.35 -> 20.15, 2048 x 2048 at 2048 53.3 -> 52.2, 4096 x 2048 at 2000 90.1 ->
// 88.0, 3000 x 2000 at 3000 98.7 -> 96.3; 512 x 2048 at 4096 29.26 -> 29.38.  Not wide tiles (2048 x 8192 at 4096 247.2 -> 248.6, at 2500
// 200.3 -> 201.6; their dW launch alone 199.8).
constexpr int BESIDE = 1, AHEAD = 2;

struct KParams {
  int M, N, Kc;
  int bn;                 // tile width
  int stages, stage_bytes;   // ring depth, bytes of a stage (both CTAs alike)
  int splits;             // CTA pairs that share a tile's contraction: 1, or 2 / 4 (one tile per cluster then)
  int n_main;             // WIDE: columns of the second accumulator half (the first has 256); otherwise
                          // tile columns of bn; a last column with at most bn/2 columns of the matrix (narrow) is extra
  int narrow;             // 1: there is such a column; its tiles are bn/2 wide
  int n_full;             // the first n_full tiles of the main columns are bn wide, the others come as two halves (tail split)
  uint32_t* status;
  long long ext_yout, ext_dyt, ext_state, ext_wsoft;   // bytes of Yout, dYt, each of V / m / u / dV, wsoft_next (debug checks)
  // REF / FWD
  void* Yout; int yout_dtype; long long ldy;
  const void* Yref; int yref_dtype;
  int columns;            // REF: Yout is [N, ldy], the accumulator's rows are its columns (compiled in: COLUMNS); FWD, BWD: 0, BESIDE or AHEAD
  int yref_t;             // FWD: Y_ref / Y_q stored transposed, [O, ldy] with ldy >= T rounded up to 16; REF: rows of Yout are
                          // padded like that, columns beyond N up to the next multiple of 16 are written as 0
  int y_store;            // REF: rows of Yout take 2: 32-byte stores, 1: 16-byte stores, 0: single values
  __nv_bfloat16* dYt; long long ld_dyt;
  float mse2c;
  float act_scale;        // FWD: Y_q = act_scale * acc; BWD: G = act_scale * acc
  float* partials;
  // BWD: M = O, N = K
  Segment seg[FAAR_MAX_SEGMENTS];
  int seg_end[FAAR_MAX_SEGMENTS - 1];   // first rows of segments 1 and 2
  // constants of the update, derived once on the host: as kernel parameters they are operands of the instructions that
  // use them and take no registers
  float bl, hbl;                    // beta log2(e) (e^x as 2^(x log2 e)), -bl / 2
  float sbeta;                      // beta act_scale / 2 (the narrowest interval is 0.5 wide)
  float b1, b2, c1, c2, eps;        // c = 1 - b
  float nstep;                      // -lr / bias correction 1 (Adam), -lr (gradient descent)
  float rbc2;                       // sqrt(u / bc2) = sqrt(u) rbc2
  float nbl_next, hbl_next;         // the next step's Eq. 3 (faar_operand_consts)
  // BWD, optional: the next step's BF16 forward operand, from the updated v (null = not wanted)
  __nv_bfloat16* wsoft_next;
  // BWD, optional: the CTA that finishes last also forms the step's two loss values (see the end of the kernel)
  unsigned long long* fin_word;     // workspace word, zero between launches
  double fin_unit, fin_inv_unit;    // fixed-point units per 1 of the Round Loss sum, a power of two; its inverse
  unsigned long long* fin_far;      // workspace: one bit per CTA whose sum does not fit the fixed-point field (zero between launches)
  double* fin_far_sums;             // and those sums, by CTA
  const float* fin_mse_partials; int fin_n_mse; float fin_scale_mse;
  float fin_scale_round; float* fin_out2;   // {L_MSE, L_round}; null = no final sums here
  long long ext_partials;           // bytes of partials: loss sums, softmax statistics or row sums (debug checks)
};

// Tile t of the launch: the first n_full tiles of the raster are bn wide, each of the others is taken as two tiles of
// bn/2 (half-width tiles even out the last, partly empty wave of the CTA pairs and halve the epilogue that
// nothing overlaps).  All full-width tiles come first.  Tiles are numbered in bands of RASTER_ROWS row blocks, inside
// a band row block fastest: the tiles that run at one time (74) then form a nearly square patch of the output, which
// needs the fewest distinct operand rows.  With row blocks fastest over the whole height the LM head's product
// (128 256 x 8192 outputs, 501 row blocks) read its 525 MB of weights from DRAM once per token tile.
constexpr int RASTER_ROWS = 8;
struct TileCoord { int m0, n0, w; };
__device__ __forceinline__ void raster(int t, int m_tiles, int n_cols, int& m, int& n) {
  const int band = t / (RASTER_ROWS * n_cols), first = band * RASTER_ROWS;
  const int rows = min(RASTER_ROWS, m_tiles - first), r = t - first * n_cols;
  n = r / rows;
  m = first + r - n * rows;
}
__device__ __forceinline__ TileCoord tile_coord(const KParams& p, int t, int m_tiles) {
  const int halves = 2 * (m_tiles * p.n_main - p.n_full);
  const int u = t - p.n_full;
  TileCoord c;
  int m, n;
  if (u < halves) {
    raster(u < 0 ? t : p.n_full + (u >> 1), m_tiles, p.n_main, m, n);
    c.n0 = n * p.bn + (u > 0 ? (u & 1) * (p.bn / 2) : 0);
    c.w = u < 0 ? p.bn : p.bn / 2;
  } else {
    m = u - halves;
    c.n0 = p.n_main * p.bn;
    c.w = p.bn / 2;
  }
  c.m0 = m * (2 * BM);
  return c;
}
__device__ __forceinline__ int tile_count(const KParams& p, int m_tiles) {
  return 2 * m_tiles * p.n_main - p.n_full + (p.narrow ? m_tiles : 0);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&p);
}

// Debug build (-DFAAR_DEBUG): every epilogue store is checked against the extent of the tensor it writes; a
// store that would leave it is skipped and recorded in the status word (0xD00 | tensor id), which
// faar_check_status reports.  No trap, no assert: the kernel runs on.  In the normal build the check is gone.
#ifdef FAAR_DEBUG
__device__ __forceinline__ bool dbg_in_range(const KParams& p, const void* ptr, long long bytes, const void* base,
                                             long long extent, uint32_t id) {
  const long long off = reinterpret_cast<const char*>(ptr) - reinterpret_cast<const char*>(base);
  if (off >= 0 && off + bytes <= extent) return true;
  atomicCAS(p.status, 0u, 0xD00u | id);
  return false;
}
#define FAAR_DBG_OK(p, ptr, bytes, base, extent, id) dbg_in_range(p, ptr, bytes, base, extent, id)
#else
#define FAAR_DBG_OK(p, ptr, bytes, base, extent, id) true
#endif

// ---- epilogues: one call handles 16 accumulator columns of one row ---------------------------
__device__ __forceinline__ void stg256(void* ptr, const uint32_t (&w)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(ptr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]),
               "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
}
// REF: write acc to row `row`, columns c0..c0+15 of Y.  A whole 32-byte sector per lane and instruction: with the output
// feature in the lane and the token in the column (2-byte stores, 64 bytes per warp instruction) the epilogue of a
// 256-wide tile took 7.4-9 us, most of it after the last product of a launch.
__device__ __forceinline__ void store_units(void* y, const uint32_t (&w)[8], bool wide) {      // 32 bytes
  if (wide) { stg256(y, w); return; }
  reinterpret_cast<uint4*>(y)[0] = make_uint4(w[0], w[1], w[2], w[3]);
  reinterpret_cast<uint4*>(y)[1] = make_uint4(w[4], w[5], w[6], w[7]);
}
// The accumulator's rows as columns of Y: neighbouring lanes write neighbouring values, whatever the alignment of a row of Y.
// A chunk's 16 stores go out together, which shortens an epilogue that nothing hides.  apart: one after the other, each behind
// its own test, where the next tile's main loop is long enough to hide that: back to back these stores of 64 bytes of a row (FP32:
// 128) get in the way of its operands.  BF16 products with 3 values of padding a row, us, together -> apart: [4000, 12288] over
// 2048 144.6 -> 141.2 (one by one everywhere, as before: 141.3), [8192, 4096] over 3072 141.1 -> 135.0 (139.0), over 1536 75.4 -> 72.7
// (75.9); over 1280 64.6 -> 64.5 (67.8) and [3000, 8192] over 1024, where every tile's stores go out together, 43.1 (50.1).  FP32
// [4000, 12288] over 1536 123.1 -> 122.0 (122.0), over 2048 154.6 either way.  Tiles of up to 128 columns gain nothing ([128,
// 128256] over 2048 87.4 -> 87.6).
constexpr int APART_BLOCKS = 24;
template <typename T>
__device__ __forceinline__ void store_columns(const KParams& p, int col, int r0, const uint32_t (&acc)[16], bool apart) {
  T* y = reinterpret_cast<T*>(p.Yout) + (long long)r0 * p.ldy + col;
  auto store = [&](int j) {
    if (!FAAR_DBG_OK(p, y + j * p.ldy, (int)sizeof(T), p.Yout, p.ext_yout, 1u)) return;
    if constexpr (sizeof(T) == 2) y[j * p.ldy] = __float2bfloat16_rn(__uint_as_float(acc[j]));
    else y[j * p.ldy] = __uint_as_float(acc[j]);
  };
  if (r0 + 16 <= p.N && !apart) {
#pragma unroll
    for (int j = 0; j < 16; ++j) store(j);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (r0 + j < p.N) store(j);
  }
}
__device__ __forceinline__ void epi_ref_columns(const KParams& p, int col, int r0, const uint32_t (&acc)[16], bool apart) {
  if (col >= p.M) return;
  if (p.yout_dtype == FAAR_BF16) store_columns<__nv_bfloat16>(p, col, r0, acc, apart);
  else store_columns<float>(p, col, r0, acc, apart);
}
// 16 columns as BF16 pairs, those beyond the matrix as 0.  One test for all of them: `whole || column < N` for each became 16
// branches, 600 clocks per 16 columns and most of a 256-wide tile's epilogue, which nothing hides for a pair's last tile:
// products over 2048, us: [2000, 2048] 18.1 -> 16.8, [2000, 4096] 28.5 -> 27.1; [2000, 2048] over 6144 38.7 -> 37.3.
__device__ __forceinline__ void pack_ref(const KParams& p, int c0, const uint32_t (&acc)[16], uint32_t (&w)[8]) {
  if (c0 + 16 <= p.N) {
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = pack_bf16x2(__uint_as_float(acc[2 * j]), __uint_as_float(acc[2 * j + 1]));
    return;
  }
  const uint32_t valid = (1u << max(p.N - c0, 0)) - 1u;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    w[j] = pack_bf16x2(valid >> (2 * j) & 1u ? __uint_as_float(acc[2 * j]) : 0.f, valid >> (2 * j + 1) & 1u ? __uint_as_float(acc[2 * j + 1]) : 0.f);
}
__device__ __forceinline__ void epi_ref(const KParams& p, int row, int c0, const uint32_t (&acc)[16]) {
  if (row >= p.M) return;
  const long long off = (long long)row * p.ldy + c0;
  const bool whole = c0 + 16 <= p.N, wide = p.y_store == 2;
  if (p.y_store && (whole || p.yref_t)) {
    if (p.yout_dtype == FAAR_BF16) {
      __nv_bfloat16* y = reinterpret_cast<__nv_bfloat16*>(p.Yout) + off;
      uint32_t w[8];
      pack_ref(p, c0, acc, w);
      if (FAAR_DBG_OK(p, y, 32, p.Yout, p.ext_yout, 1u)) store_units(y, w, wide);
    } else {
      float* y = reinterpret_cast<float*>(p.Yout) + off;
      if (!FAAR_DBG_OK(p, y, 64, p.Yout, p.ext_yout, 1u)) return;
      const uint32_t valid = whole ? 0xFFFFu : (1u << max(p.N - c0, 0)) - 1u;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t w[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) w[j] = valid >> (8 * h + j) & 1u ? acc[8 * h + j] : 0u;
        store_units(y + 8 * h, w, wide);
      }
    }
    return;
  }
  const int n = min(16, p.N - c0);
  if (p.yout_dtype == FAAR_BF16) {
    __nv_bfloat16* y = reinterpret_cast<__nv_bfloat16*>(p.Yout) + off;
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (j < n && FAAR_DBG_OK(p, y + j, 2, p.Yout, p.ext_yout, 1u)) y[j] = __float2bfloat16_rn(__uint_as_float(acc[j]));
  } else {
    float* y = reinterpret_cast<float*>(p.Yout) + off;
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (j < n && FAAR_DBG_OK(p, y + j, 4, p.Yout, p.ext_yout, 1u)) y[j] = __uint_as_float(acc[j]);
  }
}

// REF of a decoder block's gate and up projections (weights stacked, N = 2 f): a tile holds w / 2 columns of the gate and the
// same w / 2 of up, since either half of a tile's B rows is loaded by one CTA of the pair and the second one's start f rows
// further on.  A lane then has both values of its 16 features and writes act = silu(gate) up (p.dYt, rows of p.ld_dyt) next
// to them, or, where nobody reads them again (p.Yout null), instead of them: the values that a product rounded to BF16 and
// faar_silu_mul give, without that call's pass over 3 f values a token.  The main loop hides it.  Product and call -> this, us:
// 8192 tokens, f 8192 over 2048 338 + 59 -> 336 (with gate and up written too 348); 2000, 6144 over 2048 69.5 + 13.2 -> 70 (72).
// The contraction is never split here: that would part a feature's two columns.
__device__ __forceinline__ void epi_gated_fwd(const KParams& p, int row, int c0, const uint32_t (&gate)[16], const uint32_t (&up)[16]) {
  if (row >= p.M) return;
  uint32_t g[8], u[8], a[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    g[j] = pack_bf16x2(__uint_as_float(gate[2 * j]), __uint_as_float(gate[2 * j + 1]));
    u[j] = pack_bf16x2(__uint_as_float(up[2 * j]), __uint_as_float(up[2 * j + 1]));
    a[j] = pack_bf16x2(faar_silu_mul(__uint_as_float(g[j] << 16), __uint_as_float(u[j] << 16)),
                       faar_silu_mul(__uint_as_float(g[j] & 0xFFFF0000u), __uint_as_float(u[j] & 0xFFFF0000u)));
  }
  __nv_bfloat16* act = p.dYt + (long long)row * p.ld_dyt + c0;
  if (FAAR_DBG_OK(p, act, 32, p.dYt, p.ext_dyt, 2u)) stg256(act, a);
  if (!p.Yout) return;
  __nv_bfloat16* y = reinterpret_cast<__nv_bfloat16*>(p.Yout) + (long long)row * p.ldy + c0;
  if (FAAR_DBG_OK(p, y, 32, p.Yout, p.ext_yout, 1u)) stg256(y, g);
  if (FAAR_DBG_OK(p, y + p.N / 2, 32, p.Yout, p.ext_yout, 1u)) stg256(y + p.N / 2, u);
}
// REF of the input gradient of a block's down projection (N = f): the accumulator is the gradient towards act; from it and the
// gate and up values of the forward pass (p.Yref, rows as Yout's: gate, then up) come the gradients of both (p.Yout).
//
// Gate and up come in (and both gradients leave) as 16 bytes a lane, a row of 32 columns in four neighbouring lanes, the
// accumulator's columns passing through the warp's panel of shared memory for it, which fits next to the ring's six stages: a
// lane reading its own row's 32 bytes holds a line of L1 for each, and 28 KB of L1 then keep too few bytes in flight.  Sixteen
// warps, because a warp's loads, arithmetic and stores do not overlap.  Input gradient and element-wise call -> this, us: 8192
// tokens, f 8192 over 2048 167 + 108 -> 204 (lanes reading their own rows 250; eight warps of 64 columns 224); 2000, 6144 over
// 2048 40.5 + 18.6 -> 49.  More L1 for a stage of the ring (as SHORT_TILES): 212.
struct GateUp { uint4 g, u; };
struct GateRows {                                // which of the warp's 32 rows and 16-byte units a lane takes in step `it` of a panel
  int log_units;                                 // 2 or 4 units a row
  __device__ __forceinline__ int steps() const { return 1 << log_units; }
  __device__ __forceinline__ int row(int lane, int it) const { return (it << (5 - log_units)) + (lane >> log_units); }
  __device__ __forceinline__ int unit(int lane) const { return lane & ((1 << log_units) - 1); }
};
__device__ __forceinline__ uint32_t gate_unit(uint32_t panel, int row, int u) { return panel + (uint32_t)(row * 64 + ((u ^ (row >> 1 & 3)) << 4)); }
__device__ __forceinline__ void load_gate_up(const KParams& p, int row, int col, int col_end, GateUp& v) {
  if (row >= p.M || col >= col_end) return;
  const __nv_bfloat16* y = reinterpret_cast<const __nv_bfloat16*>(p.Yref) + (long long)row * p.ldy + col;
  v.g = *reinterpret_cast<const uint4*>(y);
  v.u = *reinterpret_cast<const uint4*>(y + p.N);
}
__device__ __forceinline__ void epi_gated_bwd(const KParams& p, int row, int col, int col_end, uint32_t staged, const GateUp& v) {
  if (row >= p.M || col >= col_end) return;
  const float4 raw = lds128(staged);
  const uint32_t d[4] = {__float_as_uint(raw.x), __float_as_uint(raw.y), __float_as_uint(raw.z), __float_as_uint(raw.w)};
  const uint32_t g[4] = {v.g.x, v.g.y, v.g.z, v.g.w}, u[4] = {v.u.x, v.u.y, v.u.z, v.u.w};
  uint32_t dg[4], du[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float g0, g1, u0, u1;
    faar_silu_mul_bwd(__uint_as_float(d[j] << 16), __uint_as_float(g[j] << 16), __uint_as_float(u[j] << 16), g0, u0);
    faar_silu_mul_bwd(__uint_as_float(d[j] & 0xFFFF0000u), __uint_as_float(g[j] & 0xFFFF0000u), __uint_as_float(u[j] & 0xFFFF0000u), g1, u1);
    dg[j] = pack_bf16x2(g0, g1);
    du[j] = pack_bf16x2(u0, u1);
  }
  __nv_bfloat16* y = reinterpret_cast<__nv_bfloat16*>(p.Yout) + (long long)row * p.ldy + col;
  if (FAAR_DBG_OK(p, y, 16, p.Yout, p.ext_yout, 1u)) *reinterpret_cast<uint4*>(y) = make_uint4(dg[0], dg[1], dg[2], dg[3]);
  if (FAAR_DBG_OK(p, y + p.N, 16, p.Yout, p.ext_yout, 1u)) *reinterpret_cast<uint4*>(y + p.N) = make_uint4(du[0], du[1], du[2], du[3]);
}

// REF of a block's q / k / v projections: the heads of q and k leave turned by their row's angles (p.Yref: [head_dim / 2, M]
// sines and cosines, p.yref_dtype: head_dim, p.ld_dyt: columns of q and k; tiles are whole heads).  A warp takes 16 of a head's
// head_dim / 2 angles at a time, which serve all heads of the tile; the first 16 are requested before the accumulator is
// ready.  The values of the product rounded to BF16 and faar_rope.  Product and call -> this, us:
// [8192, 3072] over 2048 69.6 + 17.4 -> 70.2, [2000, 4096] over 2048 28.9 + 8.3 -> 29.8.  (Sines and cosines formed here: 70.8 and
// 34.0; angles of a row side by side, a line of L1 per lane: 30.6.)
__device__ __forceinline__ void load_angles(const KParams& p, int row, int c, float2 (&sc)[16]) {
  if (row >= p.M || c >= p.yref_dtype / 2) return;
  const float2* t = reinterpret_cast<const float2*>(p.Yref) + (long long)c * p.M + row;
#pragma unroll
  for (int j = 0; j < 16; ++j) sc[j] = t[(long long)j * p.M];
}
__device__ __forceinline__ void store_row(const KParams& p, int row, int c0, const uint32_t (&w)[8]) {
  __nv_bfloat16* y = reinterpret_cast<__nv_bfloat16*>(p.Yout) + (long long)row * p.ldy + c0;
  if (FAAR_DBG_OK(p, y, 32, p.Yout, p.ext_yout, 1u)) stg256(y, w);
}
__device__ __forceinline__ void epi_rope(const KParams& p, uint32_t trow, int row, int n0, int width, int cg, int groups, float2 (&sc)[16]) {
  const int hd = p.yref_dtype, turning = (int)p.ld_dyt - n0, end = min(width, p.N - n0);
#pragma unroll 1
  for (int c = 16 * cg; c < hd / 2; c += 16 * groups) {
    if (c >= 16 * groups) load_angles(p, row, c, sc);
#pragma unroll 1
    for (int h = 0; h < end; h += hd) {
      uint32_t a[16], b[16], lo[8], hi[8];
      tmem_ld16(trow + (uint32_t)(h + c), a);
      tmem_ld16(trow + (uint32_t)(h + hd / 2 + c), b);
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        lo[j] = pack_bf16x2(__uint_as_float(a[2 * j]), __uint_as_float(a[2 * j + 1]));
        hi[j] = pack_bf16x2(__uint_as_float(b[2 * j]), __uint_as_float(b[2 * j + 1]));
      }
      if (h < turning) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          float x0 = __uint_as_float(lo[j] << 16), x1 = __uint_as_float(lo[j] & 0xFFFF0000u);
          float y0 = __uint_as_float(hi[j] << 16), y1 = __uint_as_float(hi[j] & 0xFFFF0000u);
          faar_rope_turn(x0, y0, sc[2 * j].x, sc[2 * j].y);
          faar_rope_turn(x1, y1, sc[2 * j + 1].x, sc[2 * j + 1].y);
          lo[j] = pack_bf16x2(x0, x1);
          hi[j] = pack_bf16x2(y0, y1);
        }
      }
      if (row < p.M) {
        store_row(p, row, n0 + h + c, lo);
        store_row(p, row, n0 + h + hd / 2 + c, hi);
      }
      __syncwarp();
    }
  }
}

// REF of an LM head's logits (whole 256-wide tiles): with the BF16 values go, per row and 128 columns, the maximum m of y = c z and the
// sum of 2^(y - m) (p.partials: [M, slots] pairs; p.mse2c: c), from which the alignment loss has a row's log-sum-exp without a pass
// of its own over the logits.  A warp's 128 columns are one slot; its lanes keep (m, s) of their rows over the 32 columns in
// registers.  Under the main loop: [8192, 128256] over 2048 2.85 ms either way, [2000, 32000] 150 us.
__device__ __forceinline__ void stats_update(const KParams& p, const uint32_t (&acc)[16], float& m, float& s) {
  float z[16];
#pragma unroll
  for (int j = 0; j < 8; ++j) {                          // as they are stored
    const uint32_t w = pack_bf16x2(__uint_as_float(acc[2 * j]), __uint_as_float(acc[2 * j + 1]));
    z[2 * j] = __uint_as_float(w << 16);
    z[2 * j + 1] = __uint_as_float(w & 0xFFFF0000u);
  }
  faar_stats_update(z, p.mse2c, m, s);
}

// Attention output's gradient dO = dY W (B untransposed): delta = sum of dO * O over a head's columns, which the attention's backward
// pass starts from, leaves with it instead of taking a launch of its own in the chain.  A lane's row of O (p.Yref, rows like Yout's)
// is asked for 32 columns ahead, the first of a tile before the wait for the accumulator.  Whatever widths the launch
// takes, a warp's columns are whole units of ld_dyt (16 .. head_dim, see launch_variant); every unit's sum is stored for itself,
// p.partials: [head_dim / unit][heads][M], and the attention kernels add them up.  Sums of 16 columns meet in a binary tree, here as
// there: the result does not depend on the widths.  The launch that it replaces -> this, alignment
// step, us: two blocks of 64-element heads on 192 tokens 195 -> 190, four on 1200 371.7 -> 366.0, two of 128-element heads on 400 264.6 ->
// 260.2; long sequences, whose launches are large, 0.3 % at most.
__device__ __forceinline__ void load_sum_row(const KParams& p, int row, int col, int end, uint4 (&v)[4]) {
  if (row >= p.M) return;
  const uint4* at = reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.Yref) + (long long)row * p.ldy + col);
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (col + 8 * q < end) v[q] = at[q];
}
__device__ __forceinline__ void sum_update(const KParams& p, int row, int col, const uint32_t (&acc)[16], const uint4& v0, const uint4& v1,
                                           float (&pending)[3]) {
  float sum = 0.f;
  const uint32_t ow[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
  for (int j = 0; j < 8; ++j) {                          // dO as it is stored
    const uint32_t w = pack_bf16x2(__uint_as_float(acc[2 * j]), __uint_as_float(acc[2 * j + 1]));
    sum = fmaf(__uint_as_float(ow[j] << 16), __uint_as_float(w << 16), sum);
    sum = fmaf(__uint_as_float(ow[j] & 0xFFFF0000u), __uint_as_float(w & 0xFFFF0000u), sum);
  }
  const int unit = (int)p.ld_dyt, dim = p.yref_dtype;    // powers of two
#pragma unroll
  for (int level = 0; level < 3; ++level) {
    if (16 << level >= unit) break;
    if (!(col >> (4 + level) & 1)) { pending[level] = sum; return; }
    sum = pending[level] + sum;
  }
  const int head = col >> (31 - __clz(dim)), part = (col & (dim - 1)) >> (31 - __clz(unit));
  float* at = p.partials + ((long long)part * (p.N >> (31 - __clz(dim))) + head) * p.M + row;
  if (row < p.M && FAAR_DBG_OK(p, at, 4, p.partials, p.ext_partials, 5u)) *at = sum;
}

// FWD: residual, sum of squares, dY^T.
// Y_ref[t0..t0+15, o] for this lane's output feature o, as it is in memory: anything done to a value here (widening BF16, a
// select at the matrix edge) would wait for it here, one latency per chunk of 16 columns.  Forward kernel, row-major target,
// before -> after: 4096 x 2048 at 2048 tokens BF16 90 -> 45, FP32 51 -> 46 us (transposed BF16: 40); 5312 x 304 at 1504
// tokens 74 -> 27 and 32 -> 26.
__device__ __forceinline__ void load_yref(const KParams& p, int o, int t0, uint32_t (&yr)[16]) {
  if (o >= p.M) return;
  const bool bf16 = p.yref_dtype == FAAR_BF16;
  if (p.yref_t) {
    if (bf16) {
      const uint4* y4 = reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.Yref) + (long long)o * p.ldy + t0);
      const uint4 a = y4[0], b = y4[1];
      yr[0] = a.x; yr[1] = a.y; yr[2] = a.z; yr[3] = a.w;
      yr[4] = b.x; yr[5] = b.y; yr[6] = b.z; yr[7] = b.w;
    } else {
      const uint4* y4 = reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(p.Yref) + (long long)o * p.ldy + t0);
#pragma unroll
      for (int q = 0; q < 4; ++q) { const uint4 v = y4[q]; yr[4 * q] = v.x; yr[4 * q + 1] = v.y; yr[4 * q + 2] = v.z; yr[4 * q + 3] = v.w; }
    }
  } else if (bf16) {
    const uint16_t* y = reinterpret_cast<const uint16_t*>(p.Yref);
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (t0 + j < p.N) asm volatile("ld.global.u16 %0, [%1];" : "=r"(yr[j]) : "l"(y + (long long)(t0 + j) * p.ldy + o));
  } else {
    const uint32_t* y = reinterpret_cast<const uint32_t*>(p.Yref);
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (t0 + j < p.N) asm volatile("ld.global.b32 %0, [%1];" : "=r"(yr[j]) : "l"(y + (long long)(t0 + j) * p.ldy + o));
  }
}
// the same as numbers (columns beyond the matrix: anything)
__device__ __forceinline__ void yref_values(const KParams& p, const uint32_t (&raw)[16], float (&yr)[16]) {
  const int shift = p.yref_dtype == FAAR_BF16 ? 16 : 0;
  const bool pairs = p.yref_t && shift;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const uint32_t pair = j & 1 ? raw[j >> 1] & 0xFFFF0000u : raw[j >> 1] << 16;
    yr[j] = __uint_as_float(pairs ? pair : raw[j] << shift);
  }
}

// Asks L2 for a warp's part of a row-major target: 32 rows of the accumulator from o_first, columns [t0, t1), one line per
// column (two where the row's start makes its values span two).
__device__ __forceinline__ void prefetch_yref(const KParams& p, int lane, int o_first, int t0, int t1) {
  if (o_first >= p.M) return;
  const long long es = p.yref_dtype == FAAR_BF16 ? 2 : 4;
  const int last = min(o_first + 31, p.M - 1);
  for (int t = t0 + lane; t < min(t1, p.N); t += 32) {
    const char* row = reinterpret_cast<const char*>(p.Yref) + (long long)t * p.ldy * es;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(row + o_first * es) : "memory");
    asm volatile("prefetch.global.L2 [%0];" ::"l"(row + last * es) : "memory");
  }
}
// 16 BF16 values of a row of dY^T: one 32-byte store where the row allows it (any token count that rounds up to 16)
__device__ __forceinline__ void store_row16(__nv_bfloat16* out, const uint32_t (&d)[8]) {
  if ((reinterpret_cast<uintptr_t>(out) & 31) == 0) {
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(out), "r"(d[0]), "r"(d[1]), "r"(d[2]), "r"(d[3]), "r"(d[4]),
                 "r"(d[5]), "r"(d[6]), "r"(d[7]) : "memory");
  } else {
    reinterpret_cast<uint4*>(out)[0] = make_uint4(d[0], d[1], d[2], d[3]);
    reinterpret_cast<uint4*>(out)[1] = make_uint4(d[4], d[5], d[6], d[7]);
  }
}

__device__ __forceinline__ float epi_fwd(const KParams& p, int o, int t0, const uint32_t (&acc)[16], const float (&yr)[16]) {
  if (o >= p.M) return 0.f;
  float ss = 0.f;
  float dy[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    float a = __uint_as_float(acc[j]) * p.act_scale;
    float r = (t0 + j < p.N) ? a - yr[j] : 0.f;
    ss = fmaf(r, r, ss);
    dy[j] = p.mse2c * r;
  }
  __nv_bfloat16* drow = p.dYt + (long long)o * p.ld_dyt + t0;
  if (!FAAR_DBG_OK(p, drow, 2 * (t0 + 16 <= p.N ? 16 : p.N - t0), p.dYt, p.ext_dyt, 2u)) return ss;
  if (t0 + 16 <= p.N) {
    uint32_t d[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) d[i] = pack_bf16x2(dy[2 * i], dy[2 * i + 1]);
    store_row16(drow, d);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (t0 + j < p.N) drow[j] = __float2bfloat16_rn(dy[j]);
  }
  if (p.Yout) {
    __nv_bfloat16* yq = reinterpret_cast<__nv_bfloat16*>(p.Yout);
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (t0 + j < p.N) {
        __nv_bfloat16* q = yq + (p.yref_t ? (long long)o * p.ldy + t0 + j : (long long)(t0 + j) * p.ldy + o);
        if (FAAR_DBG_OK(p, q, 2, p.Yout, p.ext_yout, 1u)) *q = __float2bfloat16_rn(__uint_as_float(acc[j]) * p.act_scale);
      }
  }
  return ss;
}

// The same for a chunk inside the matrix, 16 target values held as BF16 pairs (transposed target), no Y_q wanted: two
// values at a time, which keeps the whole epilogue in registers.
__device__ __forceinline__ float epi_fwd_vec(const KParams& p, int o, int t0, const uint32_t (&acc)[16], const uint4& ya, const uint4& yb) {
  if (o >= p.M) return 0.f;
  const uint32_t w[8] = {ya.x, ya.y, ya.z, ya.w, yb.x, yb.y, yb.z, yb.w};
  float ss = 0.f;
  uint32_t d[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float r0 = __uint_as_float(acc[2 * i]) * p.act_scale - __uint_as_float(w[i] << 16);
    const float r1 = __uint_as_float(acc[2 * i + 1]) * p.act_scale - __uint_as_float(w[i] & 0xFFFF0000u);
    ss = fmaf(r0, r0, ss);
    ss = fmaf(r1, r1, ss);
    d[i] = pack_bf16x2(p.mse2c * r0, p.mse2c * r1);
  }
  __nv_bfloat16* drow = p.dYt + (long long)o * p.ld_dyt + t0;
  if (!FAAR_DBG_OK(p, drow, 32, p.dYt, p.ext_dyt, 2u)) return ss;
  store_row16(drow, d);
  return ss;
}

// ---- BWD epilogue ----------------------------------------------------------------------------
__device__ __forceinline__ float sqrt_approx(float x) {       // sqrt(0) = 0, about 1 ulp
  float y;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The four epilogue warps that share a TMEM lane quarter stage a 32-row x PW-column panel of G in
// shared memory (row r at panel + 4 PW r, its 16-byte units swizzled: panel_unit); then warp `sub`
// of the quarter takes rows 8 sub .. 8 sub + 7, LPR = PX / LW lanes per row and lane l the columns
// LW (l % LPR) and on, so that one warp instruction moves 128 LW bytes of V / m / u as 32 / LPR row pieces of
// 4 PX contiguous bytes each, as 16- or 32-byte vectors: two lines (half a line or one where PX is 16 or 32).  (A panel of 128 columns gives one 512-byte
// piece per instruction but leaves room for five TMA stages only; the sixth stage is worth more.)
// The per-weight state of the next instruction is requested before the current one's is computed, and a panel's first
// before the panel is staged (a tile's first before its accumulator is ready): a request takes 600-800 clocks, the
// arithmetic of one instruction's weights about 400, and a small launch has nothing else to hide the former.
// o_first: output feature of panel row 0; k_first: input feature of panel column 0; k_end: first
// input feature beyond the tile (or the matrix).
// Returns the Round Loss contribution of the pre-update v's.
// LW is 4, or 8 in launches of short contractions (Cfg::LANE_WEIGHTS); PX the columns that the lanes of a row cover: PW, or 16
// or 32 (SPLIT_NARROW).
// 16-byte unit `u` of row `row` of a panel: the row moves its units around so that a column of rows does not collide, and with
// eight columns a lane even units lie in a row's first half, odd ones in its second, so that its lanes read consecutive units.
template <int LW> __device__ __forceinline__ uint32_t panel_unit(uint32_t panel, int row, int u) {
  return panel + (uint32_t)row * (4u * PW) + (uint32_t)((LW == 4 ? u ^ (row & 7) : ((u >> 1) ^ (row & 7)) | (u & 1) << 3) << 4);
}
template <int LW> struct RowState { float v[LW], m[LW], u[LW]; uint32_t cw, sb; };
// State of this lane's LW weights of instruction `it` of the panel whose row 0 / column 0 is (o_first, k_first), or
// nothing if they lie outside the matrix or at or beyond column k_end.
template <int OPT, int LW, int PX>
__device__ __forceinline__ bool load_row_state(const KParams& p, const Segment& g, int lane, int sub, int o_first, int k_first, int k_end, int it,
                                               uint64_t stream, RowState<LW>& st) {
  constexpr int LPR = PX / LW, RPI = 32 / LPR;                     // lanes per panel row; rows per warp instruction
  const int row = o_first + 8 * sub + lane / LPR + RPI * it, col = k_first + LW * (lane % LPR);
  const bool ok = row < p.M && col < k_end;
  if (ok) {
    const long long e = (long long)row * p.N + col;
    ldg_state(g.V + e, g.wide, stream, st.v);
    if (LW == 4) st.cw = *reinterpret_cast<const uint16_t*>(g.code + (e >> 1));
    else st.cw = *reinterpret_cast<const uint32_t*>(g.code + (e >> 1));
    st.sb = g.scales[e >> 4];
    if (OPT & 1) {
      ldg_state(g.adam_m + e, g.wide, stream, st.m);
      ldg_state(g.adam_u + e, g.wide, stream, st.u);
    }
  }
  return ok;
}
// `st` / `st_ok` hold the state of instruction 0 on entry; on return those of instruction 0 of the panel at column
// k_next (unless k_next >= k_end).
template <int OPT, int LW, int PX>
__device__ __forceinline__ float epi_bwd_rows(const KParams& p, const Segment& sg, uint32_t panel, int lane, int sub, int o_first,
                                              int k_first, int k_next, int k_end, float s_global, RowState<LW>& st, bool& st_ok) {
  constexpr int LPR = PX / LW, RPI = 32 / LPR, ITS = 8 / RPI;      // ITS: instructions per warp and panel
  const int cu = lane % LPR;                                       // LW columns of the row
  const int r0 = 8 * sub + lane / LPR;                             // this lane's row in the first instruction
  const long long e0 = (long long)(o_first + r0) * p.N + k_first + LW * cu;        // row r0 element of this lane
  const uint64_t stream = l2_policy_stream();
  const uint64_t vkeep = l2_policy_keep();       // the updated V is the next kernel's input (soft weights)
  float tt = 0.f, n_el = 0.f;                                     // sum of (2 v - 1)^2, elements seen
#pragma unroll
  for (int it = 0; it < ITS; ++it) {
    RowState<LW> cur = st;
    const bool ok = st_ok;
    st_ok = it + 1 < ITS ? load_row_state<OPT, LW, PX>(p, sg, lane, sub, o_first, k_first, k_end, it + 1, stream, st)
                         : load_row_state<OPT, LW, PX>(p, sg, lane, sub, o_first, k_next, k_end, 0, stream, st);
    if (!ok) continue;
    const int row = r0 + RPI * it;
    const long long e = e0 + (long long)(RPI * it) * p.N;
    const float sc = __fmul_rn(faar_e4m3_to_float(cur.sb), s_global);
    const float sbh = sc * p.sbeta;
    float g[LW];
    uint32_t wn[LW / 2];
#pragma unroll
    for (int h = 0; h < LW / 4; ++h) {
      const float4 g4 = lds128(panel_unit<LW>(panel, row, LW / 4 * cu + h));
      const float G[4] = {g4.x, g4.y, g4.z, g4.w};
      const uint32_t cw = h ? cur.cw >> 16 : cur.cw;
      // byte j: log2 of (interval width / 0.5) of element j, looked up by its interval index k (0 0 0 0 1 1 2)
      const uint32_t ksel = cw & 0x7777u;
      const uint32_t wlog = __byte_perm(0u, 0x00020101u, ksel);
      // OPT & 2: bytes 3 and 2 of the lower node's float (0 .5 1 1.5 2 3 4) by the same look-up
      uint32_t lo_hi = 0u, lo_lo = 0u;
      if (OPT & 2) {
        lo_hi = __byte_perm(0x3F3F3F00u, 0x00404040u, ksel);
        lo_lo = __byte_perm(0xC0800000u, 0x00804000u, ksel);
      }
      float w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float& v = cur.v[4 * h + j];
        const float ex = faar_ex2(-fabsf(fmaf(p.bl, v, p.hbl)));         // e^-|beta (v - 0.5)|
        const float hs = rcp_approx(1.0f + ex);
        const float dh = ex * hs * hs;                                     // h (1 - h)
        // dh times the width factor by an add to its exponent field (a dh flushed to 0 becomes ~1e-38), then
        // the sign of w from bit 3 of the nibble
        const uint32_t wexp = (j < 3 ? wlog << (23 - 8 * j) : wlog >> 1) & 0x01800000u;
        const uint32_t sgn = (cw << (28 - 4 * j)) & 0x80000000u;
        float chain = sbh * __uint_as_float(__float_as_uint(dh) + wexp);
        chain = __uint_as_float(__float_as_uint(chain) ^ sgn);
        const float t = fmaf(2.f, v, -1.f);
        const float gj = fmaf(G[j], chain, sg.lam4 * t);
        g[4 * h + j] = gj;
        tt = fmaf(t, t, tt);
        if (OPT & 1) {
          float &m = cur.m[4 * h + j], &u = cur.u[4 * h + j];
          m = fmaf(p.b1, m, p.c1 * gj);
          u = fmaf(p.b2, u, p.c2 * gj * gj);
          const float den = fmaf(sqrt_approx(u), p.rbc2, p.eps);
          v = __saturatef(fmaf(p.nstep, m * rcp_approx(den), v));           // clip to [0, 1]
        } else {
          v = __saturatef(fmaf(p.nstep, gj, v));
        }
        if (OPT & 2) {
          // Eq. 2 / Eq. 3 at the updated v with the next step's beta: (lo + h width) s with the sign of w, in
          // the soft-weights kernel's operations, so that the BF16 operand is the same bit for bit
          const float lo = __uint_as_float(__byte_perm(lo_hi, lo_lo, (uint32_t)((j << 12) | ((4 + j) << 8))) & 0xFFFF0000u);
          const float wd = __uint_as_float(0x3F000000u + wexp);
          const float mag = faar_operand_weight(faar_sigmoid_operand(p.nbl_next, p.hbl_next, v), lo, wd, sc);
          w[j] = __uint_as_float(__float_as_uint(mag) ^ sgn);
        }
      }
      if (OPT & 2) {
        wn[2 * h] = pack_bf16x2(w[0], w[1]);
        wn[2 * h + 1] = pack_bf16x2(w[2], w[3]);
      }
    }
    // one check covers the five stores below: they share the element offset e
    if (!FAAR_DBG_OK(p, sg.V + e, 4 * LW, sg.V, p.ext_state, 3u)) continue;
    if ((OPT & 2) && !FAAR_DBG_OK(p, p.wsoft_next + e, 2 * LW, p.wsoft_next, p.ext_wsoft, 4u)) continue;
    if (OPT & 2) {
      if constexpr (LW == 4) *reinterpret_cast<uint2*>(p.wsoft_next + e) = make_uint2(wn[0], wn[1]);
      else *reinterpret_cast<uint4*>(p.wsoft_next + e) = make_uint4(wn[0], wn[1], wn[2], wn[3]);
    }
    if (sg.dV) stg_state(sg.dV + e, sg.wide, stream, g);
    if (OPT & 1) {
      stg_state(sg.adam_m + e, sg.wide, stream, cur.m);
      stg_state(sg.adam_u + e, sg.wide, stream, cur.u);
    }
    stg_state(sg.V + e, sg.wide, vkeep, cur.v);
    n_el += (float)LW;
  }
  return n_el - tt;                                               // sum of 1 - (2 v - 1)^2
}

// ---- split contraction -----------------------------------------------------------------------
// The pairs of a cluster finish consecutive shares of the tile's columns, in whole chunks of 16: pair d those from
// share_begin(w, splits, d) on.  What arrives from the other pairs lies behind the operand ring as
// [part][4 columns][row] of 16 bytes: a warp, one row per lane, reads and writes consecutive 16-byte units.
__host__ __device__ constexpr int share_begin(int w, int splits, int d) { return 16 * ((w / 16) * d / splits); }
constexpr int largest_share(int w, int splits) { return 16 * ((w / 16 + splits - 1) / splits); }
constexpr int parts_bytes(int splits, int w) { return (splits - 1) * largest_share(w, splits) * BM * 4; }
__device__ __forceinline__ uint32_t part_unit(uint32_t parts, int slot, int cols, int unit, int row) {
  return parts + (uint32_t)(((slot * (cols >> 2) + unit) * BM + row) << 4);
}
// One epilogue warp's share of the exchange: `trow` is the warp's lane quarter of the tile's accumulator, w columns wide.
// Nobody waits before sending: the room is used once and for this alone, and the stores themselves complete the
// receiver's barrier (a handshake, fences and arrivals around plain stores took 1.4 us more).  False: the wait for the
// others' parts gave up.
__device__ __forceinline__ bool exchange_parts(uint32_t trow, int w, int splits, int split, uint32_t prank, uint32_t parts,
                                               uint32_t bar_recv, int quarter, int cg, int groups, int lane, const AbortCtl& ac) {
  const int row = quarter * 32 + lane;
  int i = 0;
  for (int d = 0; d < splits; ++d) {
    if (d == split) continue;
    const int slot = split < d ? split : split - 1, c0 = share_begin(w, splits, d), cols = share_begin(w, splits, d + 1) - c0;
    const uint32_t dst = 2u * (uint32_t)d + prank, bar = map_to_cta(bar_recv, dst);
    for (int c = 0; c < cols; c += 16, ++i) {
      if (i % groups != cg) continue;
      uint32_t r[16];
      tmem_ld16(trow + (uint32_t)(c0 + c), r);
      tmem_ld_wait();
#pragma unroll
      for (int u = 0; u < 4; ++u)
        st_async128(map_to_cta(part_unit(parts, slot, cols, (c >> 2) + u, row), dst), r[4 * u], r[4 * u + 1], r[4 * u + 2], r[4 * u + 3], bar);
    }
  }
  return __all_sync(0xffffffffu, mbar_wait_cluster(bar_recv, 0u, ac, 0x800u));
}
// r += what the other pairs sent for the 16 columns from `c` (of this pair's share, `cols` wide) of this lane's row; four
// parts as (0 + 1) + (2 + 3), which is the same sum whichever of them is the own one.
__device__ __forceinline__ void add_parts(uint32_t (&r)[16], uint32_t parts, int splits, int split, int cols, int c, int row) {
  auto slot = [&](int j) { return j < split ? j : j - 1; };
  const int other = (split ^ 2) & 2;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const float4 v = lds128(part_unit(parts, slot(split ^ 1), cols, (c >> 2) + u, row));
    const float p[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) r[4 * u + j] = __float_as_uint(__uint_as_float(r[4 * u + j]) + p[j]);
    if (splits == 4) {
      const float4 x = lds128(part_unit(parts, slot(other), cols, (c >> 2) + u, row));
      const float4 y = lds128(part_unit(parts, slot(other + 1), cols, (c >> 2) + u, row));
      const float q[4] = {x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) r[4 * u + j] = __float_as_uint(__uint_as_float(r[4 * u + j]) + q[j]);
    }
  }
}

// ---- the kernel ------------------------------------------------------------------------------
// Launched as clusters of 2 * splits CTAs along x; CTAs 2c and 2c+1 form a pair.
// MN: bit 0 = the A operand, bit 1 = the B operand is stored with its M / N index contiguous (KParams.a_mn / b_mn);
// a compile-time choice, so that the K-major kernels carry no trace of the other layout in their issue loops.  Bit 2 (REF): the
// accumulator's rows are the result's columns; compiled in as well (as a branch it cost 0.1 us in every small product).  Bit 3
// (REF): the gated product's epilogue, forward, or backward where B is N-contiguous.  Bit 4 (REF): heads turn by their position.  Bit 5
// (REF): each row's softmax statistics leave with it.  Bit 6 (REF, B untransposed): so do the row sums of the attention's gradient.
// SHAPE: one of the tile forms (see Cfg).
constexpr int MIN_SPLIT_BLOCKS = 12;            // contractions of fewer k blocks stay whole (see pick_splits)
template <int MODE, int OPT, int SHAPE, int MN>
__global__ void __launch_bounds__(Cfg<MODE, SHAPE, MN>::THREADS, 1)
faar_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ KParams p) {
  using C = Cfg<MODE, SHAPE, MN>;
  constexpr bool WIDE = C::WIDE, SPLIT = C::SPLIT;
  constexpr int LW = C::LANE_WEIGHTS;
  constexpr bool A_MN = (MN & 1) != 0, B_MN = (MN & 2) != 0, COLUMNS = (MN & 4) != 0, GATED = MN == GATED_FWD, GATED_B = MN == GATED_BWD;
  const int BN = p.bn;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;       // the same offset in both CTAs of the pair
  uint8_t* smem = smem_raw + (base - raw);
  const int STAGES = p.stages;
  const uint32_t STAGE_BYTES = (uint32_t)p.stage_bytes;
  const uint32_t epi_u32 = base + C::RING_BYTES;
  uint8_t* ctl = smem + C::RING_BYTES + C::EPI_BYTES;
  const uint32_t ctl_u32 = epi_u32 + C::EPI_BYTES;
  // control block: full[S], empty[S], tmem_full[2], tmem_empty[2], tmem base, abort flag
  auto full_bar = [&](int s) { return ctl_u32 + 8u * s; };
  auto empty_bar = [&](int s) { return ctl_u32 + 8u * (MAX_STAGES + s); };
  auto tfull_bar = [&](int a) { return ctl_u32 + 8u * (2 * MAX_STAGES + a); };
  auto tempty_bar = [&](int a) { return ctl_u32 + 8u * (2 * MAX_STAGES + 2 + a); };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(ctl + 8 * (2 * MAX_STAGES + 4));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(ctl + 8 * (2 * MAX_STAGES + 4) + 4);
  double* fin_mse = reinterpret_cast<double*>(ctl + 320);            // BWD with final sums: L_MSE's sum
  float* fin_warp = reinterpret_cast<float*>(ctl + 328);             // and the epilogue warps' Round Loss sums
  volatile int* fin_flags = reinterpret_cast<volatile int*>(ctl + 392);   // 0: a warp's sum is out of range; 1: no final sums
  const AbortCtl ac{abort_flag, p.status};

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int splits = SPLIT ? p.splits : 1;
  const uint32_t crank = cluster_ctarank();
  const uint32_t rank = SPLIT ? crank & 1u : crank, leader = SPLIT ? crank & ~1u : 0u;   // rank 0 = leader of the pair
  const int split = SPLIT ? (int)(crank >> 1) : 0;     // this pair's part of the contraction
  const int pair = blockIdx.x / (2 * splits), n_pairs = gridDim.x / (2 * splits);      // (clusters, with splits > 1)
  const int m_tiles = (p.M + 2 * BM - 1) / (2 * BM);
  // WIDE: tiles of 256 + n_main columns, numbered row block fastest; no tail split
  const int wide_w = BN_MAX + p.n_main;
  const int total_tiles = WIDE ? m_tiles * ((p.N + wide_w - 1) / wide_w) : tile_count(p, m_tiles);
  const int k_blocks = (p.Kc + BK - 1) / BK;
  const int kb0 = SPLIT ? k_blocks * split / splits : 0, kb1 = SPLIT ? k_blocks * (split + 1) / splits : k_blocks;
  const uint32_t bar_recv = ctl_u32 + 208u, parts = base + (uint32_t)STAGES * STAGE_BYTES;   // SPLIT: see exchange_parts

  if (threadIdx.x == 64) {                             // the copies' descriptors, fetched during the set-up
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    // accumulator-empty barriers are used in the leader only: every epilogue warp of both CTAs arrives there
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), 2 * C::EPI_WARPS); }
    if (SPLIT) { mbar_init(bar_recv, 1); mbar_expect_tx(bar_recv, (uint32_t)((splits - 1) * (share_begin(BN, splits, split + 1) - share_begin(BN, splits, split)) * BM * 4)); }
    for (int q = 0; q < 8; ++q) mbar_init(ctl_u32 + 256u + 8u * q, 4);   // panel staged / panel consumed, per lane quarter
    *abort_flag = 0;
    if (MODE == FAAR_GEMM_BWD) fin_flags[0] = fin_flags[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), C::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  cluster_sync_all();                                  // barriers of both CTAs are initialised
  tc_fence_after();
  // set-up done; now wait for the previous kernel's data: all of it, or (AHEAD) only the producer for the A operand
  if (MODE != FAAR_GEMM_REF && !WIDE && p.columns != 0) faar_pdl_launch();
  else if (MODE != FAAR_GEMM_BWD) faar_pdl_wait_first();
  else faar_pdl_sync();
  const uint32_t tmem_base = *tmem_slot;

  const uint64_t keep = l2_policy_keep();
  // one stage's B operand (this CTA's half); the leader's barrier collects the bytes of both CTAs' copies of A and B
  auto load_b = [&](const TileCoord& tc, int kb, int stage) {
    const int n0 = GATED ? tc.n0 / 2 + (int)rank * (p.N / 2) : tc.n0 + (int)rank * (tc.w / 2);
    const uint32_t sb = base + stage * STAGE_BYTES + C::A_BYTES, leader_full = map_to_cta(full_bar(stage), leader);
    if (rank == 0)
      mbar_expect_tx(full_bar(stage), WIDE ? 2u * (uint32_t)(C::A_BYTES + wide_w / 2 * BK * 2)
                                           : 2u * (uint32_t)(C::A_BYTES + (B_MN ? mn_boxes(tc.w / 2) * MN_BOX : tc.w / 2) * BK * 2));
    if (B_MN) {                                            // this CTA's w / 2 columns of B, in boxes of 64
      tma_load_2d(sb, &tmB, n0, kb * BK, leader_full, keep);
      if (tc.w / 2 > MN_BOX) tma_load_2d(sb + MN_BOX_BYTES, &tmB, n0 + MN_BOX, kb * BK, leader_full, keep);
    } else {
      tma_load_2d(sb, tc.w == BN ? &tmB : &tmBh, kb * BK, n0, leader_full, keep);      // box of w / 2 rows
    }
    // second column half (rows beyond the matrix arrive as zeros)
    if (WIDE) tma_load_2d(sb + C::BH_BYTES, &tmBh, kb * BK, tc.n0 + BN_MAX + (int)rank * (p.n_main / 2), leader_full, keep);
  };
  auto coords = [&](int tile) {
    TileCoord tc;
    if (WIDE) { tc.m0 = (tile % m_tiles) * (2 * BM); tc.n0 = (tile / m_tiles) * wide_w; tc.w = BN; }
    else tc = tile_coord(p, tile, m_tiles);
    return tc;
  };
  const bool b_ahead = MODE != FAAR_GEMM_REF && !WIDE && p.columns == AHEAD;      // the first ring of B is warp 1's to ask for, under the
                                                                          // end of the kernel before

  if (warp == 0) {
    // ---------------- TMA producer (both CTAs; the whole warp, converged: see faar_elect_one) ----------------
    int loaded = b_ahead ? min(STAGES, kb1 - kb0) : 0;
    if (b_ahead) faar_pdl_join();
    int stage = 0; uint32_t phase = 0;
    bool ok = true;
    for (int tile = pair; tile < total_tiles && ok; tile += n_pairs) {
      const TileCoord tc = coords(tile);
      const int m0 = tc.m0 + (int)rank * BM;
      for (int kb = kb0; kb < kb1; ++kb) {
        ok = __all_sync(0xffffffffu, mbar_wait(empty_bar(stage), phase ^ 1u, ac, 0x100u | stage));
        if (!ok) break;
        const uint32_t sa = base + stage * STAGE_BYTES;
        const uint32_t leader_full = map_to_cta(full_bar(stage), leader);
        const bool with_b = loaded == 0;
        if (!with_b) --loaded;
        if (faar_elect_one()) {
          if (with_b) load_b(tc, kb, stage);
          if (A_MN) {                                          // two boxes of 64 rows of A, each [64 k][64 m]
            tma_load_2d(sa, &tmA, m0, kb * BK, leader_full, keep);
            tma_load_2d(sa + MN_BOX_BYTES, &tmA, m0 + MN_BOX, kb * BK, leader_full, keep);
          } else {
            tma_load_2d(sa, &tmA, kb * BK, m0, leader_full, keep);
          }
        }
        __syncwarp();
        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok) {
      // give copies already in flight a bounded chance to land before the CTA exits
      const unsigned long long t0 = global_ns();
      while (global_ns() - t0 < 2000000ull) {}
    }
    if constexpr (MODE == FAAR_GEMM_BWD) {
      // the forward's share of the loss values, under the epilogue: strided double accumulation, then a tree over lanes
      if (p.fin_out2 != nullptr) {
        __syncwarp();
        if (lane == 0 && __ldcg(p.status) != 0u) fin_flags[1] = 1;
        double mse = 0.0;
#pragma unroll 8
        for (int i = lane; i < p.fin_n_mse; i += 32) mse += (double)__ldcg(p.fin_mse_partials + i);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mse += __shfl_xor_sync(0xffffffffu, mse, o);
        if (lane == 0) *fin_mse = mse;
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader CTA only; the whole warp, converged: see faar_elect_one) ----------------
    // (AHEAD, both CTAs: first the B ring.  By the producer itself, in front of its wait, it held up the A operand of CTAs that
    // start late: step of 512 x 2048 at 4096 tokens 30.2 -> 32.2 us)
    if (b_ahead) {
      const TileCoord tc = coords(pair);
      for (int i = 0; i < min(STAGES, kb1 - kb0); ++i) {
        if (faar_elect_one()) load_b(tc, kb0 + i, i);
        __syncwarp();
      }
    }
    if (rank == 0) {
      int stage = 0; uint32_t phase = 0;
      int it = 0;
      bool ok = true;
      for (int tile = pair; tile < total_tiles && ok; tile += n_pairs, ++it) {
        // WIDE: the two column halves take the place of the two accumulator buffers; both must be drained
        const int acc = WIDE ? 0 : it & 1;
        const uint32_t acc_phase = WIDE ? it & 1 : (it >> 1) & 1;
        ok = mbar_wait(tempty_bar(acc), acc_phase ^ 1u, ac, 0x200u | acc);
        if (ok && WIDE) ok = mbar_wait(tempty_bar(1), acc_phase ^ 1u, ac, 0x201u);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + acc * BN_MAX;
        const uint32_t idesc1 = WIDE ? make_idesc(p.n_main) : 0u;
        const uint32_t idesc = make_idesc(WIDE ? BN_MAX : tile_coord(p, tile, m_tiles).w, A_MN ? 1 : 0, B_MN ? 1 : 0);
        for (int kb = kb0; kb < kb1; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait(full_bar(stage), phase, ac, 0x300u | stage));
          if (!ok) break;
          tc_fence_after();
          const uint32_t sa = base + stage * STAGE_BYTES, sb = sa + C::A_BYTES;
          const uint64_t da = A_MN ? make_smem_desc_mn(sa) : make_smem_desc(sa);
          const uint64_t db = B_MN ? make_smem_desc_mn(sb) : make_smem_desc(sb);
          constexpr uint32_t ka = A_MN ? MN_KSTEP : 2u, kbs = B_MN ? MN_KSTEP : 2u;
          if (faar_elect_one()) {
#pragma unroll
            for (int k = 0; k < BK / UMMA_K; ++k) {
              // advancing 16 bf16 = 32 bytes inside the swizzled row: +2 in the 16-byte address field
              // (MN-major: 16 rows of 128 bytes further on)
              tc_mma_bf16(tmem_d, da + ka * k, db + kbs * k, idesc, (SPLIT ? kb != kb0 || k != 0 : (kb | k) != 0) ? 1u : 0u);
              if (WIDE)
                tc_mma_bf16(tmem_d + BN_MAX, da + 2u * k, make_smem_desc(sb + C::BH_BYTES) + 2u * k, idesc1,
                            (SPLIT ? kb != kb0 || k != 0 : (kb | k) != 0) ? 1u : 0u);
            }
            tc_commit_pair(empty_bar(stage), leader);          // frees this stage in both CTAs
          }
          __syncwarp();
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (ok && faar_elect_one()) {
          tc_commit_pair(tfull_bar(acc), leader);              // accumulator ready in both CTAs
          if (WIDE) tc_commit_pair(tfull_bar(1), leader);
        }
        __syncwarp();
      }
    }
  } else {
    // ---------------- epilogue (both CTAs) ----------------
    const int ew = warp - 2;
    const int quarter = warp & 3;                      // TMEM lanes this warp may read
    // REF / FWD: the warps that share a lane quarter split the tile's columns in 16-column chunks
    const int cg = ew >> 2;                            // which of the warps sharing this lane quarter
    float warp_acc = 0.f;
    float s_global = 0.f;
    if (MODE == FAAR_GEMM_BWD) s_global = *p.seg[0].s_global;
    uint32_t pn = 0;                                   // panels this quarter has staged so far
    RowState<LW> row_state;                               // BWD: state requested ahead
    bool row_ok = false;
    const bool yvec_ok = MODE == FAAR_GEMM_FWD && p.yref_t && p.yref_dtype == FAAR_BF16 && p.Yout == nullptr;
    bool dead = false;
    // One pass per accumulator buffer that fills: a tile, or (WIDE) a 256-column half of a tile.
    int vt = 0;
    for (;; ++vt) {
      const int it = WIDE ? vt >> 1 : vt;
      const int tile = pair + it * n_pairs;
      if (tile >= total_tiles) break;
      const int acc = WIDE ? vt & 1 : it & 1;
      const uint32_t acc_phase = WIDE ? it & 1 : (it >> 1) & 1;
      // whether a later tile takes this accumulator buffer: else nobody waits for its release
      const bool again = tile + (WIDE ? 1 : 2) * n_pairs < total_tiles;
      TileCoord tc;
      if (WIDE) { tc.m0 = (tile % m_tiles) * (2 * BM); tc.n0 = (tile / m_tiles) * wide_w + acc * BN_MAX; tc.w = acc ? p.n_main : BN_MAX; }
      else tc = tile_coord(p, tile, m_tiles);
      // the columns of the tile that this pair finishes: with a split contraction its share
      const int share0 = SPLIT ? share_begin(tc.w, splits, split) : 0;
      const int TW = SPLIT ? share_begin(tc.w, splits, split + 1) - share0 : tc.w, m0 = tc.m0 + (int)rank * BM, n0 = tc.n0 + share0;
      const int cols_per_warp = ((TW / C::COL_GROUPS + 15) / 16) * 16;
      const int col_begin = cg * cols_per_warp;
      const int col_end = min(col_begin + cols_per_warp, TW);
      const int o = m0 + quarter * 32 + lane;
      // FWD with a transposed BF16 target, columns inside the matrix: this lane's target values (128 at most, sixteen
      // 16-byte loads) are requested before the wait for the accumulator, so their latency lies under the main loop (of a
      // wide tile's second half: behind the first half's stores.  Asked for between those stores, the forward kernel and soft
      // weights of 2048 x 8192 take, us, at 4608 tokens 121.5 -> 122.3, at 4096 112.3 -> 112.9, of 4096 x 8192 at 2048 135.3 -> 136.3;
      // both halves' before the main loop, in 64 more registers, spill: 123.0, 113.7, 136.5)
      const bool yvec = yvec_ok && n0 + col_end <= p.N;
      uint4 yraw[MODE == FAAR_GEMM_FWD ? 16 : 1];
      if constexpr (MODE == FAAR_GEMM_FWD) {
        static_assert(BN_MAX / C::COL_GROUPS == 128, "a warp's columns of the widest tile");
        if (yvec && o < p.M) {
          const uint4* y4 = reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p.Yref) +
                                                           (long long)o * p.ldy + n0 + col_begin);
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (col_begin + 16 * q < col_end) { yraw[2 * q] = y4[2 * q]; yraw[2 * q + 1] = y4[2 * q + 1]; }
        }
      }
      // FWD otherwise: the target values of the warp's first 16 columns (the others one chunk ahead of their use)
      uint32_t ynext[MODE == FAAR_GEMM_FWD ? 16 : 1];
      if constexpr (MODE == FAAR_GEMM_FWD) {
        if (!yvec && col_begin < col_end && n0 + col_begin < p.N) load_yref(p, o, n0 + col_begin, ynext);
        // the others of a row-major target into L2 (5312 x 304 at 1504 tokens, tiles of 256: 27.9 -> 26.1 us; 64-wide tiles
        // have one chunk more only and lose 0.2 us by asking)
        if (!p.yref_t && col_end - col_begin > 32) prefetch_yref(p, lane, m0 + quarter * 32, n0 + col_begin + 16, n0 + col_end);
      }
      const int k_end = min(p.N, n0 + TW);               // BWD: columns of this tile that exist
      // the linear this warp's 8 rows belong to (several only with both operands row-major)
      const int o_warp = m0 + quarter * 32 + 8 * (ew >> 2);
      const Segment& seg = p.seg[MODE == FAAR_GEMM_BWD && MN == 3 ? (o_warp >= p.seg_end[0]) + (o_warp >= p.seg_end[1]) : 0];
      if constexpr (MODE == FAAR_GEMM_BWD) {
        if (MN == 3) s_global = *seg.s_global;
        const int o0 = m0 + quarter * 32;
        if constexpr (SHAPE == SPLIT_NARROW)
          row_ok = TW <= 16 ? load_row_state<OPT, LW, 16>(p, seg, lane, ew >> 2, o0, n0, k_end, 0, l2_policy_stream(), row_state)
                            : load_row_state<OPT, LW, 32>(p, seg, lane, ew >> 2, o0, n0, k_end, 0, l2_policy_stream(), row_state);
        else
          row_ok = load_row_state<OPT, LW, PW>(p, seg, lane, ew >> 2, o0, n0, k_end, 0, l2_policy_stream(), row_state);
      }
      // backward of the gated product: gate and up values of the warp's first 32 columns
      GateUp ahead[GATED_B ? 4 : 1];
      const GateRows gr = {cols_per_warp <= 16 ? 1 : 2};
      const int o_quarter = m0 + quarter * 32, gate_end = min(n0 + col_end, p.N);
      if constexpr (GATED_B) {
#pragma unroll
        for (int it = 0; it < 4; ++it)
          if (it < gr.steps()) load_gate_up(p, o_quarter + gr.row(lane, it), n0 + col_begin + 8 * gr.unit(lane), gate_end, ahead[it]);
      }
      float2 angles[MN == ROPE ? 16 : 1];
      if constexpr (MN == ROPE) load_angles(p, o, 16 * cg, angles);
      uint4 sum_row[MN == SUMS ? 4 : 1];
      const int sum_end = min(n0 + col_end, p.N);
      if constexpr (MN == SUMS) load_sum_row(p, o, n0 + col_begin, sum_end, sum_row);
      bool ok = mbar_wait(tfull_bar(acc), acc_phase, ac, 0x400u | acc);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t ttile = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * BN_MAX);
      const uint32_t trow = ttile + (uint32_t)share0;
      if (SPLIT) {
        ok = exchange_parts(ttile, tc.w, splits, split, rank, parts, bar_recv, quarter, ew >> 2, C::COL_GROUPS, lane, ac);
        if (!ok) break;
        tc_fence_after();
      }
      if constexpr (MODE == FAAR_GEMM_BWD) {
        // PW-column panels, staged by the four warps of this lane quarter together (see epi_bwd_rows)
        const int sub = ew >> 2;
        const uint32_t panel = epi_u32 + (uint32_t)quarter * PANEL_BYTES;
        const uint32_t pfull = ctl_u32 + 256u + 16u * quarter, pdone = pfull + 8u;
        const int o_first = m0 + quarter * 32;
        bool released = false;
#pragma unroll 1
        for (int pc = 0; pc < TW; pc += PW) {
          if (n0 + pc >= p.N || o_first >= p.M) break;   // the same decision in all four warps
          // the quarter's previous panel has been consumed by all four warps
          bool okp = mbar_wait(pdone, (pn & 1u) ^ 1u, ac, 0x500u | quarter);
          if (!__all_sync(0xffffffffu, okp)) { dead = true; break; }
          static_assert(PW == 64, "each of the four warps stages PW / 4 = 16 accumulator columns");
          const int c = pc + 16 * sub;
          if (c < TW && n0 + c < p.N) {
            uint32_t r[16];
            tmem_ld16(trow + (uint32_t)c, r);
            tmem_ld_wait();
            if (SPLIT) add_parts(r, parts, splits, split, TW, c, quarter * 32 + lane);
#pragma unroll
            for (int u = 0; u < 4; ++u)
              sts128(panel_unit<LW>(panel, lane, 4 * sub + u), r[4 * u], r[4 * u + 1], r[4 * u + 2], r[4 * u + 3]);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(pfull);
          if (pc + PW >= TW || n0 + pc + PW >= p.N) {    // this warp's last read of the accumulator
            tc_fence_before();
            __syncwarp();
            if (again && lane == 0) mbar_arrive_cluster(map_to_cta(tempty_bar(acc), leader));
            released = true;
          }
          okp = mbar_wait(pfull, pn & 1u, ac, 0x600u | quarter);
          if (!__all_sync(0xffffffffu, okp)) { dead = true; break; }
          const int k0 = n0 + pc, k1 = k0 + PW;            // SPLIT_NARROW: one panel
          if constexpr (SHAPE == SPLIT_NARROW)
            warp_acc += TW <= 16 ? epi_bwd_rows<OPT, LW, 16>(p, seg, panel, lane, sub, o_first, k0, k1, k_end, s_global, row_state, row_ok)
                                 : epi_bwd_rows<OPT, LW, 32>(p, seg, panel, lane, sub, o_first, k0, k1, k_end, s_global, row_state, row_ok);
          else
            warp_acc += epi_bwd_rows<OPT, LW, PW>(p, seg, panel, lane, sub, o_first, k0, k1, k_end, s_global, row_state, row_ok);
          __syncwarp();
          if (lane == 0) mbar_arrive(pdone);
          ++pn;
        }
        if (dead) break;
        if (!released) {
          tc_fence_before();
          __syncwarp();
          if (again && lane == 0) mbar_arrive_cluster(map_to_cta(tempty_bar(acc), leader));
        }
        continue;
      } else if constexpr (GATED_B) {
        const uint32_t panel = epi_u32 + (uint32_t)(ew * GATE_PANEL);
#pragma unroll 1
        for (int c0 = col_begin; c0 < col_end && n0 + c0 < p.N; c0 += GATE_COLS) {
#pragma unroll
          for (int q = 0; q < GATE_COLS / 16; ++q) {
            const int c = c0 + 16 * q;
            if (c < col_end) {                           // warp-uniform
              uint32_t r[16];
              tmem_ld16(trow + (uint32_t)c, r);
              tmem_ld_wait();
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                uint32_t w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = pack_bf16x2(__uint_as_float(r[8 * h + 2 * j]), __uint_as_float(r[8 * h + 2 * j + 1]));
                sts128(gate_unit(panel, lane, 2 * q + h), w[0], w[1], w[2], w[3]);
              }
            }
          }
          __syncwarp();
          const int col = n0 + c0 + 8 * gr.unit(lane);
#pragma unroll
          for (int it = 0; it < 4; ++it) {
            if (it < gr.steps()) {
              const int row = o_quarter + gr.row(lane, it);
              epi_gated_bwd(p, row, col, gate_end, gate_unit(panel, gr.row(lane, it), gr.unit(lane)), ahead[it]);
              load_gate_up(p, row, col + GATE_COLS, gate_end, ahead[it]);
            }
          }
          __syncwarp();
        }
      } else if constexpr (MN == ROPE) {
        epi_rope(p, trow, o, n0, tc.w, cg, C::COL_GROUPS, angles);
      } else if constexpr (GATED) {
        // the warps of a lane quarter take 16 features of the tile in turn
        const int half = tc.w / 2, f0 = n0 / 2;
#pragma unroll 1
        for (int c = 16 * cg; c < half && f0 + c < p.N / 2; c += 16 * C::COL_GROUPS) {
          uint32_t r[16], r2[16];
          tmem_ld16(trow + (uint32_t)c, r);
          tmem_ld16(trow + (uint32_t)(half + c), r2);
          tmem_ld_wait();
          epi_gated_fwd(p, o, f0 + c, r, r2);
          __syncwarp();
        }
      } else {
        if (MODE == FAAR_GEMM_FWD && yvec) {
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int c = col_begin + 16 * q;
            if (c < col_end) {                           // warp-uniform
              uint32_t r[16];
              tmem_ld16(trow + (uint32_t)c, r);
              tmem_ld_wait();
              warp_acc += epi_fwd_vec(p, o, n0 + c, r, yraw[2 * q], yraw[2 * q + 1]);
              __syncwarp();
            }
          }
        } else {
          // REF: two chunks' accumulators in flight (a warp's column count is a multiple of 16: the second may be absent)
          constexpr int STEP = MODE == FAAR_GEMM_REF ? 32 : 16;
          float sm = -INFINITY, ssum = 0.f;              // STATS
          float pending[3];                              // SUMS
          const bool apart = COLUMNS && BN > 128 && k_blocks >= APART_BLOCKS && tile + n_pairs < total_tiles;
#pragma unroll 1
          for (int c = col_begin; c < col_end; c += STEP) {
            if (n0 + c >= p.N) break;                    // warp-uniform
            uint32_t r[16];
            tmem_ld16(trow + (uint32_t)c, r);
            if constexpr (MODE == FAAR_GEMM_REF) {
              const bool second = c + 16 < col_end && n0 + c + 16 < p.N;
              uint32_t r2[16];
              if (second) tmem_ld16(trow + (uint32_t)(c + 16), r2);
              tmem_ld_wait();
              if (SPLIT) {
                add_parts(r, parts, splits, split, TW, c, quarter * 32 + lane);
                if (second) add_parts(r2, parts, splits, split, TW, c + 16, quarter * 32 + lane);
              }
              if (COLUMNS) {
                epi_ref_columns(p, o, n0 + c, r, apart);
                if (second) epi_ref_columns(p, o, n0 + c + 16, r2, apart);
              } else {
                epi_ref(p, o, n0 + c, r);
                if (second) epi_ref(p, o, n0 + c + 16, r2);
                if constexpr (MN == STATS) {
                  stats_update(p, r, sm, ssum);
                  if (second) stats_update(p, r2, sm, ssum);
                }
                if constexpr (MN == SUMS) {
                  sum_update(p, o, n0 + c, r, sum_row[0], sum_row[1], pending);
                  if (second) sum_update(p, o, n0 + c + 16, r2, sum_row[2], sum_row[3], pending);
                  load_sum_row(p, o, n0 + c + 32, sum_end, sum_row);
                }
              }
            } else {
              float yr[16];
              yref_values(p, ynext, yr);
              if (c + 16 < col_end && n0 + c + 16 < p.N) load_yref(p, o, n0 + c + 16, ynext);
              tmem_ld_wait();
              warp_acc += epi_fwd(p, o, n0 + c, r, yr);
            }
            __syncwarp();
          }
          if constexpr (MN == STATS) {
            const int slots = (p.N + 127) / 128, slot = (n0 + col_begin) / 128;
            float2* at = reinterpret_cast<float2*>(p.partials) + (long long)o * slots + slot;
            if (o < p.M && n0 + col_begin < p.N && FAAR_DBG_OK(p, at, 8, p.partials, p.ext_partials, 5u)) *at = make_float2(sm, ssum);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (again && lane == 0) mbar_arrive_cluster(map_to_cta(tempty_bar(acc), leader));
    }
    if (MODE == FAAR_GEMM_FWD || (MODE == FAAR_GEMM_BWD && p.fin_out2 != nullptr)) {
      warp_acc = faar_warp_sum(warp_acc);
      if (lane == 0) {
        if (MODE == FAAR_GEMM_FWD) {
          float* at = p.partials + blockIdx.x * C::EPI_WARPS + ew;
          if (FAAR_DBG_OK(p, at, 4, p.partials, p.ext_partials, 5u)) *at = warp_acc;
        } else {
          fin_warp[ew] = warp_acc;
          // one per weight that the warp may have had
          const int columns = SPLIT ? share_begin(BN, splits, split + 1) - share_begin(BN, splits, split) : BN;
          if (!(fabsf(warp_acc) <= (float)(vt * (BM * columns / C::EPI_WARPS)))) fin_flags[0] = 1;
        }
      }
    }
  }

  __syncwarp();
  // No CTA may leave while another one can still read its shared memory, write its tensor memory or arrive on its
  // barriers.  Whatever one CTA does to another's has been waited for there by now (operands and accumulators: by the
  // accumulator-full barrier; releases nobody waits for are not sent), so this only has to keep the CTAs together: a
  // relaxed arrival, which does not wait until this CTA's results have reached L2 (the end of the kernel waits for that
  // anyway; about 0.5 us per launch: a small layer's step 17.2 -> 16.4, of 1000 x 1040 22.6 -> 21.3).
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) cluster_arrive_release();
  else asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (*abort_flag) {                                   // a wait gave up: what others sent here may still be on its way
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < 2000000ull) {}
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }

  if constexpr (MODE == FAAR_GEMM_BWD) {
    if (p.columns == BESIDE && threadIdx.x == 0) faar_pdl_join();
    // Final loss sums by whichever CTA finishes last.  Each adds its Round Loss sum to one word, as a fixed-point number
    // above nine bits that count the CTAs and nine that count sums kept elsewhere.  A sum is rounded to the field's unit
    // (2^-20 for 16 M weights); the addition is exact, so neither the order nor which CTA is last matters, and the last one
    // has the total from that one atomic (a small layer's step 18.1 -> 17.2 us, of 1000 x 1040 24.5 -> 22.6 against partials
    // in memory that it had to read back).  The field has room for one per weight of every CTA's tiles, which is what v in
    // [0, 1] can give.  A sum beyond that (v outside, infinite or not a number) goes to the CTA's slot in memory with a bit
    // that says so; the last CTA adds those in the order of the CTAs.  After a wait that gave up this CTA's sums are
    // incomplete: it does not count, so nobody forms final sums (the caller re-initialises the workspace, which also clears
    // the word and the bits).  Nor does anybody if an earlier launch's status is set: the forward's sums may be incomplete.
    if (p.fin_out2 != nullptr && threadIdx.x == 0 && !*abort_flag && !fin_flags[1]) {
      double rnd = 0.0;
#pragma unroll
      for (int w = 0; w < C::EPI_WARPS; ++w) rnd += (double)fin_warp[w];
      constexpr uint32_t COUNT = (1u << FIN_COUNT_BITS) - 1u;
      unsigned long long mine = ((unsigned long long)__double2ll_rn(rnd * p.fin_unit) << (2 * FIN_COUNT_BITS)) + 1ull;
      if (fin_flags[0]) {
        p.fin_far_sums[blockIdx.x] = rnd;
        atomicOr(p.fin_far + (blockIdx.x >> 6), 1ull << (blockIdx.x & 63));
        __threadfence();
        mine = 1ull + (1ull << FIN_COUNT_BITS);
      }
      const unsigned long long sum = atomicAdd(p.fin_word, mine) + mine;
      if (((uint32_t)sum & COUNT) == gridDim.x) {
        *p.fin_word = 0ull;                                  // ready for the next launch
        double total = (double)((long long)sum >> (2 * FIN_COUNT_BITS)) * p.fin_inv_unit;
        if (((uint32_t)sum >> FIN_COUNT_BITS & COUNT) != 0u) {
          __threadfence();
          for (uint32_t c = 0; c < gridDim.x; ++c)
            if (__ldcg(p.fin_far + (c >> 6)) >> (c & 63) & 1ull) total += __ldcg(p.fin_far_sums + c);
          for (uint32_t i = 0; i <= (gridDim.x - 1) >> 6; ++i) p.fin_far[i] = 0ull;
        }
        p.fin_out2[0] = (float)(*fin_mse * (double)p.fin_scale_mse);
        p.fin_out2[1] = (float)(total * (double)p.fin_scale_round);
      }
    }
  }
}

// A wait that nothing will ever satisfy, with a short limit: exercises the give-up path of the bounded
// waits (status word, flag, orderly exit) without any other kernel machinery.
__global__ void __launch_bounds__(64, 1) wait_selftest_kernel(uint32_t* status, unsigned long long limit_ns) {
  __shared__ alignas(8) unsigned long long bar;
  __shared__ int flag;
  const uint32_t b = smem_u32(&bar);
  if (threadIdx.x == 0) {
    mbar_init(b, 1);
    flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  AbortCtl ac{&flag, status, limit_ns};
  if (threadIdx.x == 0) (void)mbar_wait(b, 0u, ac, 0x700u);       // nobody arrives: gives up after limit_ns
  __syncthreads();
  if (threadIdx.x == 32) (void)mbar_wait(b, 0u, ac, 0x701u);      // sees the raised flag and leaves at once
}

// ---- host side ----------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// rows x cols bf16 matrix, cols contiguous, row stride ld elements; box = box_rows x 64.
int make_map(faar_ctx* ctx, CUtensorMap* map, const void* ptr, int rows, int cols, int64_t ld, int box_rows) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = reinterpret_cast<EncodeTiledFn>(ctx->encode_tiled)(
      map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : (int)cudaErrorInvalidValue;
}

// An operand stored [kc_rows, mn_cols] (M or N contiguous, row stride ld elements): boxes of 64 x 64.
int make_map_mn(faar_ctx* ctx, CUtensorMap* map, const void* ptr, int kc_rows, int mn_cols, int64_t ld) {
  cuuint64_t dims[2] = {(cuuint64_t)mn_cols, (cuuint64_t)kc_rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)MN_BOX, (cuuint32_t)BK};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = reinterpret_cast<EncodeTiledFn>(ctx->encode_tiled)(
      map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : (int)cudaErrorInvalidValue;
}

// Tile width for an M x N output over k_blocks blocks of the contraction.  While 256-wide tiles give every CTA pair one,
// they win: a tile's time is set by the operand bytes it pulls through the SM, and the A rows are the same for any
// width.  A smaller problem is a matter of latency: its tiles run at once, each brings its share of the epilogue, and
// narrower tiles spread that over more SMs.
// REF, FWD: the width with the smallest estimated time of the busiest pair (microseconds).  A k block costs the ring's
// latency, or what the L2 needs for all pairs' operands (about 14 TB/s); the epilogue per 64 columns 0.4 (REF), 0.6 (FWD with
// a transposed BF16 target) or 0.9 (FWD otherwise); a further wave of tiles 1.
// Measured (width before -> after): product [260, 1024] over 512 8.8 -> 6.2 us (128 -> 32), forward kernel of a
// 128 x 256 layer at 1024 tokens 12.8 -> 10.7 us, input gradient [192, 128] over 384 11.1 -> 8.9 us.
// BWD: its per-weight epilogue is bound by instruction issue and a tile of it has a fixed cost of several microseconds,
// so only 128-wide tiles (cut into halves of 64 by pick_full while pairs are idle) while fewer than half of the
// pairs would have a 256-wide one; 32-wide tiles: dW kernel of a 128 x 256 layer 19.2 -> 18.8 us, of a 1024 x 3600 layer
// 33.6 -> 51 us.
int pick_bn(const faar_ctx* ctx, int mode, int M, int N, int k_blocks, int pairs, bool b_mn, bool fwd_vec) {
  if (ctx->tune_bn >= 128 && ctx->tune_bn <= BN_MAX && ctx->tune_bn % 16 == 0)
    return b_mn ? (ctx->tune_bn + 31) / 32 * 32 : ctx->tune_bn;      // a CTA's first column of an N-contiguous B: 32-byte aligned
  const long long m_tiles = (M + 2 * BM - 1) / (2 * BM);
  if (mode == FAAR_GEMM_BWD) {
    if (N <= 128 || 2 * m_tiles * ((N + BN_MAX - 1) / BN_MAX) < pairs) return 128;
    return N < BN_MAX ? (N + 31) / 32 * 32 : BN_MAX;
  }
  const int widest = N > 128 ? (N < BN_MAX ? (N + 31) / 32 * 32 : BN_MAX) : (N > 64 ? 128 : (N > 32 ? 64 : 32));
  if (m_tiles * ((N + widest - 1) / widest) >= pairs) return widest;
  const double epi64 = mode == FAAR_GEMM_FWD ? (fwd_vec ? 0.6 : 0.9) : 0.4;
  int best = widest;
  double best_cost = 1e30;
  for (int bn = widest; bn >= 32; bn = bn > 128 ? 128 : bn / 2) {
    const long long tiles = m_tiles * ((N + bn - 1) / bn);
    const long long waves = (tiles + pairs - 1) / pairs, active = tiles < pairs ? tiles : pairs;
    const double l2 = 2.0 * active * (BM + bn / 2) * BK * 2 / 1.4e7;
    const double latency = bn > 128 ? 0.22 : (bn > 64 ? 0.19 : 0.16);
    const double loop = k_blocks * (l2 > latency ? l2 : latency), epi = epi64 * bn / 64.0;
    const double cost = waves * loop + epi + (waves - 1) * (1.0 + (epi > loop ? epi - loop : 0.0));
    if (cost < best_cost - 1e-9) { best_cost = cost; best = bn; }
  }
  return best;
}

// Over how many CTA pairs a tile's contraction is split, and how wide the tiles are then.  With few tiles the time is that
// of one pair's main loop, 0.18 us per k block whatever the tile's width (a block's latency through the ring), while other
// pairs idle; parts of the contraction run at once, for an exchange of about 1 us.  Two or four parts, tiles of 64 or 128
// columns (wider ones never won: more to exchange, more to finish), as long as the device holds a cluster for every tile;
// 64-wide tiles are paid back from 12 k blocks on (two parts of them from 14), 128-wide ones, with twice the exchange,
// from 20, and from 40 four parts of those are better than two of 64.
// Measured, whole tiles -> split (parts x width), us: dW kernel of 256 x 1024 at 1024 tokens (16 k blocks) 10.0 -> 9.2
// (2 x 64), 10.0 (4 x 128), 10.3 (2 x 128); 128 x 256 at 1024 9.8 -> 8.5 (4 x 64); 128 x 1536 at 1536 (24) 11.8 -> 10.2
// (2 x 64); 300 x 2048 at 2048 14.0 -> 12.7 (2 x 128); product [128, 768] over 768 (12) 6.1 -> 5.5 (4 x 64), [1024, 83] over
// 3600 16.2 -> 9.6.
// The forward product and the frozen target are never split: their difference, the residual, is rounded to BF16, and
// it is small against either, so that another order of the sums (with the target, another rounding to BF16) moves single
// entries of the first moments by as much as their mean size.  In the dW and plain products it moves results by 1e-5.
// The choice depends on the problem and the device alone, not on forced tile widths or operand layouts, because it is part
// of the order in which an output element is summed (with M and N exchanged a plain product is split alike).
int pick_splits(int mode, int M, int N, int k_blocks, const int (&clusters)[FAAR_CLUSTER_SIZES], int* bn_out) {
  auto tiles = [](int m, int n, int bn) { return (long long)((m + 2 * BM - 1) / (2 * BM)) * ((n + bn - 1) / bn); };
  struct Form { int size, bn, least; };
  const Form four64 = {2, 64, MIN_SPLIT_BLOCKS}, two64 = {1, 64, 14}, four128 = {2, 128, 20}, two128 = {1, 128, 20};
  const bool lots = k_blocks >= 40;
  for (const Form& f : {four64, lots ? four128 : two64, lots ? two64 : four128, two128}) {
    long long n = tiles(M, N, f.bn);
    if (mode == FAAR_GEMM_REF && tiles(N, M, f.bn) > n) n = tiles(N, M, f.bn);
    if (n > clusters[f.size] || k_blocks < f.least) continue;
    *bn_out = f.bn;
    return 1 << f.size;
  }
  return 1;
}

// How many tiles of the raster stay whole.  Tiles go to CTA pairs round-robin, all whole tiles first.  A half tile costs
// 0.75 of a whole one (its A rows are loaded all the same), and the epilogue of a pair's last tile is not overlapped by
// anything (0.4 of that tile's cost).  Returns the number that minimises the busiest pair's time (ties: fewer halves).
// A pair's load depends on how many whole and how many half tiles it gets, which change only at two pair numbers.
// Cutting single tiles instead of whole tile columns matters for tall grids, whose columns hold many tiles: [8192, 2048]
// over 8192 is 256 tiles of 256 on 74 pairs, 3.46 waves: 212 us with no column worth cutting, 191 us with 34 tiles cut.
int pick_full(faar_ctx* ctx, int mode, int m_tiles, int n_main, int narrow, int bn, int pairs) {
  const int main = m_tiles * n_main, tail = narrow ? m_tiles : 0;
  if (bn % 32 != 0 || bn <= 32) return main;
  if (ctx->tune_tail >= 0) {
    const long long cut = (long long)(ctx->tune_tail > narrow ? ctx->tune_tail - narrow : 0) * m_tiles;
    return cut < main ? main - (int)cut : 0;
  }
  if (mode != FAAR_GEMM_BWD && main + tail <= pairs) return main;        // the width was chosen for this case (pick_bn)
  for (const auto& k : ctx->split_plans)
    if (k.mode == mode && k.m_tiles == m_tiles && k.n_main == n_main && k.narrow == narrow && k.bn == bn) return k.full;
  double best = -1.0;
  int best_full = main;
  const int least = main > 2 * pairs ? main - 2 * pairs : 0;
  for (int full = main; full >= least; --full) {
    const int total = 2 * main - full + tail;
    double worst = 0.0;
    const int cand[3] = {0, full % pairs, total % pairs};
    for (int p : cand) {
      if (p >= total) continue;
      const int nt = (total - p + pairs - 1) / pairs, nf = full > p ? (full - p + pairs - 1) / pairs : 0;
      const double last = nt > nf ? 0.75 : 1.0, load = nf + 0.75 * (nt - nf) + 0.4 * last;
      if (load > worst) worst = load;
    }
    if (best < 0.0 || worst < best - 1e-9) { best = worst; best_full = full; }
  }
  auto& slot = ctx->split_plans[ctx->next_plan++ % FAAR_SPLIT_PLANS];
  slot = {mode, m_tiles, n_main, narrow, bn, best_full};
  return best_full;
}

// The width of a launch's 256 x (288 .. 512) tiles (see Cfg), 0 for none.  512 on request (ctx->tune_wide == 1) wherever the
// shape allows.  They move up to a quarter less operand data, but nothing overlaps their epilogue, and they give a wave of tiles no
// halves to even it out.  Plain product of 256-wide tiles -> 512-wide, us: 80 tiles (40 wide ones) over 2048 21.6 -> 30.0; 128
// over 2048 34.0 -> 38.4, over 4096 58.0 -> 62.4, over 8192 97 -> 99; 144 over 8192 101.3 -> 100.8; forward kernel and soft
// weights of 2048 x 4096 at 4096 tokens 72.3 -> 74.2, with an FP32 target of 2048 x 8192 152 -> 164.  By themselves therefore
// only for a forward product with a transposed BF16 target and 8192 or more contraction elements, where the least width
// that gives one wave (a multiple of 16) is at most 512 and takes less main loop than the waves of 256-wide tiles: a
// sixteenth less if it leaves more than a seventh of the pairs idle, as a thin second wave of 256-wide tiles has the L2 to itself.
// Forward kernel and soft weights over 8192, 256-wide -> this, us: 2048 outputs, 4096 tokens (464 columns, 72 of 74 pairs) 116.2 ->
// 112.3, 2500 (288) 98.4 -> 87.4, 4600 (512) 124.1 -> 122.6; 7680 outputs (60 pairs), 900 tokens (464) 167.0 -> 164.3; but
// 1024 (512) 167.4 -> 170.5, and 4864 outputs (57), 1410 (480 for two waves) 139.4 -> 141.5, 1320 (448 for 1.75) 132.6 -> 135.5.
int pick_wide(faar_ctx* ctx, int mode, int M, int N, int k_blocks, int bn, int pairs, bool fwd_vec) {
  if (bn != BN_MAX || ctx->tune_wide == 0) return 0;
  if (ctx->tune_wide == 1) return (mode == FAAR_GEMM_REF && M > N ? M : N) > BN_MAX ? WIDE_BN : 0;    // REF may have either index as its rows
  if (mode != FAAR_GEMM_FWD || !fwd_vec || k_blocks < 128 || N <= BN_MAX || ctx->tune_tail >= 0 || ctx->tune_bn != 0) return 0;
  const int m_tiles = (M + 2 * BM - 1) / (2 * BM), cols = pairs / m_tiles;
  if (cols == 0) return 0;
  int w = ((N + cols - 1) / cols + 15) / 16 * 16;
  if (w <= BN_MAX || w > WIDE_BN) return 0;
  if (w < WIDE_BN_MIN) w = WIDE_BN_MIN;
  // 256-wide tiles: waves of whole ones, and a last wave, of half tiles (0.75 each, pick_full) where the pairs suffice for
  // them; a last column of up to 128 comes as half tiles anyway
  const int whole = m_tiles * (N / BN_MAX + (N % BN_MAX > BN_MAX / 2)), narrow = N % BN_MAX != 0 && N % BN_MAX <= BN_MAX / 2 ? m_tiles : 0;
  const int rest = whole % pairs;
  const double last = rest + narrow == 0 ? 0.0 : (2 * rest + narrow <= pairs ? 0.75 : (rest + narrow <= pairs ? 1.0 : 1.75));
  const double limit = (whole / pairs + last) * BN_MAX;
  const int wide_cols = (N + w - 1) / w;
  return 7 * m_tiles * wide_cols >= 6 * pairs ? (w <= limit ? w : 0) : (w < limit * 15 / 16 ? w : 0);
}

template <int MODE, int OPT, int SHAPE, int MN>
int launch_variant(faar_ctx* ctx, const faar_gemm_args* a, KParams& kp, int* n_partials_out, int bn, int max_pairs,
                   const cudaLaunchConfig_t& base_cfg) {
  using C = Cfg<MODE, SHAPE, MN>;
  constexpr bool WIDE = C::WIDE, SPLIT = C::SPLIT;
  static_assert(C::MIN_STAGES >= 3, "ring too short");
  static_assert(C::SMEM_BYTES <= SMEM_LIMIT, "shared memory budget");
  static_assert(C::EPI_WARPS <= MAX_EPI_WARPS, "partials budget");
  auto kern = faar_gemm_kernel<MODE, OPT, SHAPE, MN>;
  int e = faar_allow_smem(ctx, (const void*)kern, C::SMEM_BYTES, C::SHORT ? SHORT_CARVEOUT : -1);
  if (e) return e;
  cudaLaunchConfig_t cfg = base_cfg;
  cfg.dynamicSmemBytes = C::SMEM_BYTES;
  cfg.blockDim = dim3(C::THREADS, 1, 1);
  kp.bn = bn;
  kp.stage_bytes = WIDE ? C::STAGE_BYTES : C::A_BYTES + (a->b_mn ? mn_boxes(bn / 2) * MN_BOX_BYTES : (int)faar_align_up((size_t)(bn / 2) * BK * 2, 1024));   // whole swizzle atoms
  const int ring = (C::RING_BYTES - (SPLIT ? parts_bytes(kp.splits, bn) : 0)) / kp.stage_bytes;
  kp.stages = ring < MAX_STAGES ? ring : MAX_STAGES;
  const int m_tiles = (a->M + 2 * BM - 1) / (2 * BM), n_cols = (a->N + bn - 1) / bn;
  const int wide_w1 = kp.n_main, wide_w = BN_MAX + wide_w1, wide_cols = (a->N + wide_w - 1) / wide_w;
  const bool halves = MN != STATS && (MN != ROPE || bn / 2 % a->head_dim == 0);       // a half-width tile, too, is whole heads
  kp.narrow = (SHAPE == PLAIN_TILES || SHAPE == SHORT_TILES) && halves && bn % 32 == 0 && bn > 32 && a->N - (n_cols - 1) * bn <= bn / 2;
  kp.n_main = WIDE ? wide_w1 : n_cols - kp.narrow;
  if (MODE == FAAR_GEMM_BWD) {
    // the widest unit at which the Round Loss field holds one per weight of the tiles (half tiles counted as whole: twice
    // that) with its sign
    const long long area = (long long)m_tiles * 2 * BM * (WIDE ? wide_cols * (long long)wide_w : (long long)n_cols * bn);
    int int_bits = 1;
    while (area >> int_bits) ++int_bits;
    kp.fin_unit = ldexp(1.0, 62 - 2 * FIN_COUNT_BITS - int_bits); kp.fin_inv_unit = 1.0 / kp.fin_unit;
  }
  kp.n_full = WIDE ? 0 : (SPLIT || !halves ? m_tiles * kp.n_main : pick_full(ctx, MODE, m_tiles, kp.n_main, kp.narrow, bn, max_pairs));
  if constexpr (MN == SUMS) {
    // the widest unit of which a warp's columns are a multiple, whatever tile (or share of a split one) it has
    int unit = a->sum_dim;
    auto fit = [&](int w) {
      const int per_warp = (w / C::COL_GROUPS + 15) / 16 * 16;
      while (w % unit || per_warp % unit) unit /= 2;
    };
    if (SPLIT) unit = 16;
    else {
      fit(bn);
      if (kp.narrow || kp.n_full < m_tiles * kp.n_main) fit(bn / 2);
    }
    kp.Yref = a->sum_with; kp.yref_dtype = a->sum_dim; kp.ld_dyt = unit; kp.partials = a->sums;
    *a->sum_parts = a->sum_dim / unit;
  }
  CUtensorMap tmA, tmB, tmBh;
  e = a->a_mn ? make_map_mn(ctx, &tmA, a->A, a->Kc, a->M, a->lda) : make_map(ctx, &tmA, a->A, a->M, a->Kc, a->lda, BM);
  if (e) return e;
  if (a->b_mn) {
    e = make_map_mn(ctx, &tmB, a->B, a->Kc, a->N, a->ldb);    // one map serves full and half-width tiles
    tmBh = tmB;
  } else {
    e = make_map(ctx, &tmB, a->B, a->N, a->Kc, a->ldb, bn / 2);
    if (e) return e;
    if (WIDE) e = make_map(ctx, &tmBh, a->B, a->N, a->Kc, a->ldb, wide_w1 / 2);           // the second half's
    else if (kp.narrow || kp.n_full < m_tiles * kp.n_main) e = make_map(ctx, &tmBh, a->B, a->N, a->Kc, a->ldb, bn % 32 == 0 ? bn / 4 : bn / 2);   // half-width tiles
    else tmBh = tmB;
  }
  if (e) return e;
  const long long tiles = WIDE ? (long long)m_tiles * wide_cols
                               : 2ll * m_tiles * kp.n_main - kp.n_full + (kp.narrow ? m_tiles : 0);
  const int pairs = SPLIT ? (int)tiles * kp.splits : (int)(tiles < max_pairs ? tiles : max_pairs);
  cfg.gridDim = dim3(2 * pairs, 1, 1);
  if (n_partials_out) *n_partials_out = 2 * pairs * C::EPI_WARPS;
  ctx->last_gemm_bn = WIDE ? WIDE_BN : bn;                   // (the form; a tile may have fewer columns)
  ctx->last_gemm_pairs = pairs;
  // in columns' worth of tiles
  ctx->last_gemm_split = WIDE ? 0 : kp.narrow + (m_tiles * kp.n_main - kp.n_full + m_tiles - 1) / m_tiles;
  faar_prof_scope ps(ctx, MODE == FAAR_GEMM_REF ? FAAR_K_GEMM_REF : (MODE == FAAR_GEMM_FWD ? FAAR_K_GEMM_FWD : FAAR_K_GEMM_BWD));
  cudaError_t ce = cudaLaunchKernelEx(&cfg, kern, tmA, tmB, tmBh, kp);
  if (ce != cudaSuccess) return (int)ce;
  return (int)cudaGetLastError();
}

template <int MODE, int OPT, int MN>
int launch_tiles(faar_ctx* ctx, const faar_gemm_args* a, KParams& kp, int* n_partials_out, int bn, int max_pairs, const cudaLaunchConfig_t& cfg) {
  if constexpr (MODE != FAAR_GEMM_FWD) {
    if constexpr (MODE == FAAR_GEMM_BWD) {
      if (kp.splits > 1 && largest_share(bn, kp.splits) <= 32)
        return launch_variant<MODE, OPT, SPLIT_NARROW, MN>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
    }
    if (kp.splits > 1) return launch_variant<MODE, OPT, SPLIT_TILES, MN>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
  }
  if constexpr (MODE == FAAR_GEMM_BWD) {
    if (bn == BN_MAX && (a->Kc + BK - 1) / BK <= SHORT_BLOCKS)
      return launch_variant<MODE, OPT, SHORT_TILES, MN>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
  }
  return launch_variant<MODE, OPT, PLAIN_TILES, MN>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
}

template <int MODE, int OPT = 0>
int launch(faar_ctx* ctx, const faar_gemm_args* a, KParams& kp, int* n_partials_out) {
  using C = Cfg<MODE>;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.blockDim = dim3(C::THREADS, 1, 1);
  cfg.dynamicSmemBytes = C::SMEM_BYTES;
  cfg.stream = ctx->stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  auto kern = faar_gemm_kernel<MODE, OPT, PLAIN_TILES, 0>;               // every variant takes one CTA per SM
  const int e = faar_allow_smem(ctx, (const void*)kern, C::SMEM_BYTES);
  if (e) return e;
  const int slot = MODE == FAAR_GEMM_BWD ? 2 + OPT : MODE;
  const int max_pairs = faar_max_clusters(ctx, slot, 0, (const void*)kern, &cfg);
  const int k_blocks = (a->Kc + BK - 1) / BK;
  kp.splits = 1;
  int split_bn = BN_MAX;
  // (forced tail splits and wide tiles compare forms of the whole contraction)
  if (MODE != FAAR_GEMM_FWD && k_blocks >= MIN_SPLIT_BLOCKS && !a->whole && ctx->tune_tail < 0 && ctx->tune_wide < 0) {
    int clusters[FAAR_CLUSTER_SIZES] = {max_pairs};
    for (int i = 1; i < FAAR_CLUSTER_SIZES; ++i) {
      attr[0].val.clusterDim.x = 2u << i;
      clusters[i] = faar_max_clusters(ctx, slot, i, (const void*)kern, &cfg);
    }
    kp.splits = pick_splits(MODE, a->M, a->N, k_blocks, clusters, &split_bn);
    attr[0].val.clusterDim.x = 2u * (unsigned)kp.splits;
  }
  const bool fwd_vec = a->yref_t && a->yref_dtype == FAAR_BF16 && !a->Yout;
  int bn = pick_bn(ctx, MODE, a->M, a->N, k_blocks, max_pairs, a->b_mn != 0, fwd_vec);
  if (kp.splits > 1 && ctx->tune_bn == 0) bn = split_bn;
  const int wide = pick_wide(ctx, MODE, a->M, a->N, k_blocks, bn, max_pairs, fwd_vec);
  kp.n_main = wide > BN_MAX ? wide - BN_MAX : BN_MAX;
  const int mn = (a->a_mn ? 1 : 0) | (a->b_mn ? 2 : 0);
  if constexpr (MODE == FAAR_GEMM_REF) {
    if (a->gated == FAAR_GATED_FWD) {                   // either half of a whole or half-width tile is a multiple of 16
      if (bn != 32) bn = (bn + 63) / 64 * 64;
      return launch_variant<MODE, OPT, PLAIN_TILES, GATED_FWD>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
    }
    if (a->stats) return launch_variant<MODE, OPT, PLAIN_TILES, STATS>(ctx, a, kp, n_partials_out, BN_MAX, max_pairs, cfg);
    if (a->rope) {                                  // whole heads
      bn = (bn + a->head_dim - 1) / a->head_dim * a->head_dim;
      return launch_variant<MODE, OPT, PLAIN_TILES, ROPE>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
    }
    if (a->gated == FAAR_GATED_BWD) return launch_variant<MODE, OPT, PLAIN_TILES, GATED_BWD>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
  }
  // which operand layouts a mode is ever launched with: the plain product with B untransposed (input gradient; A, if the
  // accumulator's rows are the result's columns), the dW product with B or with both untransposed
  if constexpr (MODE == FAAR_GEMM_REF) {
    if (kp.columns && mn == 0) {
      if (kp.splits == 1 && wide)
        return launch_variant<MODE, OPT, WIDE_TILES, 4>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
      return launch_tiles<MODE, OPT, 4>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
    }
    if (kp.columns && mn == 1) return launch_tiles<MODE, OPT, 5>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
    if (mn == 2 && a->sums) return launch_tiles<MODE, OPT, SUMS>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
    if (mn == 2) return launch_tiles<MODE, OPT, 2>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
  } else if constexpr (MODE == FAAR_GEMM_BWD) {
    if (mn == 2) return launch_tiles<MODE, OPT, 2>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
    if (mn == 3) return launch_tiles<MODE, OPT, 3>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
  }
  if (mn != 0) return (int)cudaErrorInvalidValue;
  if (kp.splits == 1 && wide)
    return launch_variant<MODE, OPT, WIDE_TILES, 0>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
  return launch_tiles<MODE, OPT, 0>(ctx, a, kp, n_partials_out, bn, max_pairs, cfg);
}

}  // namespace

// Which index of a plain product Y[M, N] lies on the accumulator's rows.  N (Y's columns) where Y's rows are not 16-byte
// aligned, because neighbouring lanes then write neighbouring values instead of one lane a row of single ones: [1000, 5000]
// over 2048 with 5003 values a row 106 -> 28 us.  And N up to 128 rows of Y, which is half a tile: the tile's other half
// would be padding that is staged all the same.  M on the accumulator's rows -> N, us: 1 row of 8192 over 2048 15.1 -> 10.6,
// 64 rows 12.8 -> 12.0, 128 rows 13.1 -> 12.2, 160 rows 13.1 -> 13.8; input gradient of 8 rows of 8192 over 2048 14.5 -> 11.9.
static bool result_columns(const faar_gemm_args* a) {
  if (a->yref_t || a->gated || a->rope || a->stats || a->sums) return false;
  const long long row = a->ldy * (a->yout_dtype == FAAR_BF16 ? 2 : 4);
  return a->M <= BM || row % 16 != 0 || (reinterpret_cast<uintptr_t>(a->Yout) & 15) != 0;
}

// Which products leave statistics at all: those where every CTA pair has 256-wide tiles anyway (and more than a half-empty row
// block); a smaller one is better cut into narrower tiles.
static long long wide_tiles(int T, int vocab) { return (long long)((T + 2 * BM - 1) / (2 * BM)) * ((vocab + BN_MAX - 1) / BN_MAX); }
bool faar_logit_stats_fit(const faar_ctx* ctx, int T, int vocab) { return T > BM && wide_tiles(T, vocab) >= ctx->num_sms / 2; }
// And where they save time: such a product has no half-width tiles to even out its last wave, which both passes pay for, and the
// loss gains with the tokens.  Both forward passes of one block, 2048 wide, and the loss, without statistics -> with them, us:
// tokens x vocabulary 129 x 128256 344 -> 361, 150 x 20480 187 -> 191, 200 x 25600 197 -> 204, 256 x 50000 243 -> 247, 300 x 12800 193
// -> 198, 300 x 32000 245 -> 248, 600 x 6400 (75 tiles) 203 -> 206, 1000 x 4864 (76) 243 -> 243; 512 x 16000 223 -> 216, 600 x 9600 220 ->
// 211, 600 x 128256 786 -> 786, 1000 x 9600 272 -> 267, 2000 x 2560 311 -> 302, 2000 x 32000 667 -> 663, 4096 x 8192 728 -> 674.
bool faar_logit_stats_pays(const faar_ctx* ctx, int T, int vocab) {
  return T >= 1000 ? faar_logit_stats_fit(ctx, T, vocab) : T >= 512 && 3 * wide_tiles(T, vocab) >= 2 * ctx->num_sms;
}

int faar_launch_wait_selftest(faar_ctx* ctx, uint32_t* status, unsigned long long limit_ns) {
  wait_selftest_kernel<<<1, 64, 0, ctx->stream>>>(status, limit_ns);
  return (int)cudaGetLastError();
}

int faar_gemm_max_partials(const faar_ctx* ctx, int, int) { return ctx->num_sms * MAX_EPI_WARPS; }

int faar_launch_gemm(faar_ctx* ctx, const faar_gemm_args* args, int* n_partials_out) {
  faar_gemm_args swapped;
  const faar_gemm_args* a = args;
  KParams kp;
  kp.columns = args->mode == FAAR_GEMM_REF ? result_columns(args) : (args->beside ? BESIDE : (args->ahead ? AHEAD : 0));
  if (args->mode == FAAR_GEMM_REF && kp.columns) {
    swapped = *args;
    swapped.M = args->N; swapped.N = args->M;
    swapped.A = args->B; swapped.lda = args->ldb; swapped.a_mn = args->b_mn;
    swapped.B = args->A; swapped.ldb = args->lda; swapped.b_mn = args->a_mn;
    a = &swapped;
  }
  if (a->gated) {                                      // unsplit, f a multiple of 16, every row on 32 bytes
    const int f = a->gated == FAAR_GATED_FWD ? a->N / 2 : a->N;
    const uintptr_t at = reinterpret_cast<uintptr_t>(a->Yout) | reinterpret_cast<uintptr_t>(a->act) | reinterpret_cast<uintptr_t>(a->gate_up);
    if (a->mode != FAAR_GEMM_REF || !a->whole || f % 16 || a->ldy % 16 || at & 31 || a->a_mn || (a->b_mn != 0) != (a->gated == FAAR_GATED_BWD) ||
        a->yout_dtype != FAAR_BF16 || (a->gated == FAAR_GATED_FWD ? !a->act || a->N % 2 : !a->Yout || !a->gate_up))
      return (int)cudaErrorInvalidValue;
  }
  if (a->stats && (a->mode != FAAR_GEMM_REF || !a->whole || a->a_mn || a->b_mn || a->gated || a->rope || a->yref_t || a->N % 16 || a->ldy % 8 ||
                   (reinterpret_cast<uintptr_t>(a->Yout) & 15) || (reinterpret_cast<uintptr_t>(a->stats) & 7) || a->yout_dtype != FAAR_BF16))
    return (int)cudaErrorInvalidValue;
  if (a->rope && (a->mode != FAAR_GEMM_REF || !a->whole || a->a_mn || a->b_mn || a->gated || (a->head_dim != 64 && a->head_dim != 128) ||
                      a->N % a->head_dim || (reinterpret_cast<uintptr_t>(a->rope) & 7) || a->rope_cols % a->head_dim || a->ldy % 16 || (reinterpret_cast<uintptr_t>(a->Yout) & 31) ||
                      a->yout_dtype != FAAR_BF16))
    return (int)cudaErrorInvalidValue;
  if (a->sums && (a->mode != FAAR_GEMM_REF || a->a_mn || !a->b_mn || a->gated || a->rope || a->stats || a->yref_t || (a->sum_dim != 64 && a->sum_dim != 128) ||
                  a->N % a->sum_dim || a->ldy % 8 || ((reinterpret_cast<uintptr_t>(a->Yout) | reinterpret_cast<uintptr_t>(a->sum_with)) & 15) ||
                  !a->sum_with || !a->sum_parts || a->yout_dtype != FAAR_BF16))
    return (int)cudaErrorInvalidValue;
  kp.M = a->M; kp.N = a->N; kp.Kc = a->Kc; kp.bn = BN_MAX; kp.n_main = kp.narrow = kp.n_full = 0; kp.status = a->status;
  {
    const long long ysz = a->yout_dtype == FAAR_BF16 ? 2 : 4;
    // the last row ends after its last valid (or padded) column; REF and the transposed FWD layout: [M, ldy], else [N(T), ldy]
    const bool rows_m = (a->mode == FAAR_GEMM_REF && !kp.columns) || a->yref_t;
    kp.ext_yout = a->Yout ? (rows_m ? ((long long)(a->M - 1) * a->ldy + (a->yref_t ? (a->N + 15) / 16 * 16 : a->N))
                                    : ((long long)(a->N - 1) * a->ldy + a->M)) * ysz : 0;
    const bool al32 = a->ldy * ysz % 32 == 0 && (reinterpret_cast<uintptr_t>(a->Yout) & 31) == 0;
    const bool al16 = a->ldy * ysz % 16 == 0 && (reinterpret_cast<uintptr_t>(a->Yout) & 15) == 0;
    kp.y_store = al32 ? 2 : (al16 ? 1 : 0);
    kp.ext_dyt = a->dYt ? ((long long)(a->M - 1) * a->ld_dyt + a->N) * 2 : 0;
    kp.ext_state = (long long)a->M * a->N * 4;
    kp.ext_wsoft = (long long)a->M * a->N * 2;
    kp.ext_partials = a->stats ? (long long)a->M * ((a->N + 127) / 128) * (long long)sizeof(float2)
                               : (a->sums ? (long long)a->M * (a->N / 16) * 4 : FAAR_MAX_PARTIALS * 4ll);
  }
  kp.Yout = a->Yout; kp.yout_dtype = a->yout_dtype; kp.ldy = a->ldy;
  kp.Yref = a->Yref; kp.yref_dtype = a->yref_dtype; kp.yref_t = a->yref_t;
  kp.dYt = a->dYt; kp.ld_dyt = a->ld_dyt; kp.mse2c = a->mse2c; kp.act_scale = a->act_scale; kp.partials = a->partials;
  if (a->stats) { kp.partials = reinterpret_cast<float*>(a->stats); kp.mse2c = a->stats_c; }
  if (a->rope) {
    kp.Yref = a->rope; kp.yref_dtype = a->head_dim; kp.ld_dyt = a->rope_cols;
  }
  if (a->gated == FAAR_GATED_FWD) {
    kp.dYt = reinterpret_cast<__nv_bfloat16*>(a->act); kp.ld_dyt = a->N / 2;
    kp.ext_dyt = (long long)a->M * a->N;
  } else if (a->gated == FAAR_GATED_BWD) {
    kp.Yref = a->gate_up;
    kp.ext_yout = ((long long)(a->M - 1) * a->ldy + 2ll * a->N) * 2;
  }
  if (a->mode == FAAR_GEMM_BWD) {
    long long row0 = 0;
    for (int i = 0; i < FAAR_MAX_SEGMENTS; ++i) {
      Segment& k = kp.seg[i];
      if (i >= a->n_seg) {
        k = Segment();
        if (i) kp.seg_end[i - 1] = 0x7FFFFFFF;
        continue;
      }
      const faar_bwd_state& g = a->seg[i];
      const long long e0 = row0 * a->N;
      if (i) kp.seg_end[i - 1] = (int)row0;
      k.V = g.V - e0; k.code = g.code - e0 / 2; k.scales = g.scales - e0 / 16; k.s_global = g.s_global;
      k.adam_m = g.adam_m ? g.adam_m - e0 : nullptr; k.adam_u = g.adam_u ? g.adam_u - e0 : nullptr; k.dV = g.dV ? g.dV - e0 : nullptr;
      k.lam4 = -4.f * g.lam_over_n;
      k.wide = ((reinterpret_cast<uintptr_t>(g.V) | reinterpret_cast<uintptr_t>(g.adam_m) | reinterpret_cast<uintptr_t>(g.adam_u) |
                 reinterpret_cast<uintptr_t>(g.dV)) & 31) == 0;
      row0 += g.rows;
    }
  }
  kp.bl = a->beta * 1.44269504088896341f; kp.hbl = -0.5f * kp.bl;
  kp.sbeta = 0.5f * a->beta * a->act_scale;
  kp.b1 = a->b1; kp.b2 = a->b2; kp.c1 = 1.f - a->b1; kp.c2 = 1.f - a->b2; kp.eps = a->eps;
  kp.nstep = a->opt == 1 ? -(a->lr * a->inv_bc1) : -a->lr;
  kp.rbc2 = sqrtf(a->inv_bc2);
  kp.nbl_next = -(a->beta_next * 1.4426950408889634f); kp.hbl_next = -0.5f * kp.nbl_next;
  kp.wsoft_next = a->wsoft_next;
  kp.fin_word = a->fin_word;
  kp.fin_far = a->fin_far; kp.fin_far_sums = a->fin_far_sums;
  if (a->fin_out2 && ctx->num_sms >= 1 << FIN_COUNT_BITS) return (int)cudaErrorInvalidValue;
  kp.fin_mse_partials = a->fin_mse_partials; kp.fin_n_mse = a->fin_n_mse;
  kp.fin_scale_mse = a->fin_scale_mse; kp.fin_scale_round = a->fin_scale_round; kp.fin_out2 = a->fin_out2;
  // the BWD epilogue forms row offsets of up to 7 rows in 32-bit element counts (the entry points refuse
  // such a K with FAAR_ERR_SHAPE before they get here)
  if (a->mode == FAAR_GEMM_BWD && (long long)a->N * 8 > 0x7FFFFFFFll) return (int)cudaErrorInvalidValue;

  switch (a->mode) {
    case FAAR_GEMM_REF: return launch<FAAR_GEMM_REF>(ctx, a, kp, n_partials_out);
    case FAAR_GEMM_FWD: return launch<FAAR_GEMM_FWD>(ctx, a, kp, n_partials_out);
    case FAAR_GEMM_BWD:
      // OPT bit 0: Adam; bit 1: also write the next step's forward operand
      if (a->wsoft_next)
        return a->opt == 1 ? launch<FAAR_GEMM_BWD, 3>(ctx, a, kp, n_partials_out)
                           : launch<FAAR_GEMM_BWD, 2>(ctx, a, kp, n_partials_out);
      return a->opt == 1 ? launch<FAAR_GEMM_BWD, 1>(ctx, a, kp, n_partials_out)
                         : launch<FAAR_GEMM_BWD, 0>(ctx, a, kp, n_partials_out);
  }
  return (int)cudaErrorInvalidValue;
}
