// NVFP4 x NVFP4 GEMM on the block-scaled tensor-core path of sm_100a: consumes what the library's own
// hardening (faar_harden_pack + faar_swizzle_scales) and activation quantiser (faar_act_fakequant +
// faar_swizzle_scales) produce -- packed E2M1 codes, E4M3 block scales in the 128 x 4 tiled order, FP32 tensor
// scales -- and returns C = alpha * A B^T in BF16 ("Hardening and Inference": the final weights are
// deployable on NVFP4 hardware as they are).
//
//   C[M,N] = (sA sB) * sum_k  A[m,k] B[n,k]        A: [M, K/2] bytes, B: [N, K/2] bytes, two codes per byte
//
// A cluster of two CTAs computes a 256 x BN tile (tcgen05.mma kind::mxf4nvf4 cta_group::2, block size 16, K = 64
// per instruction, FP32 accumulators in tensor memory): CTA r loads rows 128 r .. of the A tile, its half of the B
// tile's rows, its own A scales and ALL of the tile's B scales (each CTA's half of the MMA reads them from its own
// tensor memory).  A stage of the operand ring holds 256 elements of the contraction: rows of 128 bytes by TMA
// (128-byte swizzle: 256 codes are exactly one swizzle row) and the scale tiles, 512 bytes per 128 rows x 64
// elements, by TMA too (a 3-D map over the tiled layout; tiles beyond the matrix arrive as zeros).  The leader's
// MMA warp moves a stage's scale tiles into tensor memory (tcgen05.cp, 32 lanes x 128 bits replicated to the four
// lane quarters, in both CTAs) in front of the stage's four MMAs; stages alternate between two sets of scale
// columns, so the copies of a stage do not wait for the previous stage's MMAs.
//   warp 0: producer     warp 1: tensor memory + MMA issue (leader)     warps 2-9: epilogue
// Two accumulators.  BN = 256: 512 columns do not hold two of them next to the scale columns, so the second starts
// at column 160 and shares 96 columns with the first; the epilogue drains those first and says so, and the next
// tile's MMAs wait for that only.
// What bounds it: operand bytes from L2.  C[4096, 2048], K = 8192, four operand sets in turn: 103 us for the 128 x 128
// single-CTA tiles this replaces, 71 us with the pair tile issued under `if (lane == 0)`, 33.8 us issued by an elected
// lane of a converged warp, 31 us with the MMAs left out.  A 256 x 256 pair tile needs 76 KB per 256 contraction
// elements; the widest tile has the fewest operand bytes per flop, so BN = 128 is taken only when 256-wide tiles would
// leave CTA pairs without one (see pick_wide4).  (Scale tiles written by four more warps with tcgen05.st: 69-75 us.)
// Every barrier wait is bounded (status word, orderly exit), as in the BF16 kernels.
#include <cuda.h>

#include "faar_internal.cuh"

namespace {

constexpr int TM = 128;                      // accumulator rows per CTA; the pair covers 256
constexpr int KS = 256;                      // contraction elements per stage = 128 bytes per row
constexpr int KI = 64;                       // contraction elements per MMA
constexpr int ROW_BYTES = KS / 2;            // 128
constexpr int SF_TILE = 512;                 // scales of 128 rows x 64 contraction elements
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 32 * (2 + EPI_WARPS);
constexpr int TMEM_COLS = 512;
constexpr int CTL = 256;

template <int BN> struct Cfg4 {
  static constexpr int A_BYTES = TM * ROW_BYTES;             // 16 KB
  static constexpr int B_BYTES = (BN / 2) * ROW_BYTES;       // this CTA's half of the B rows
  static constexpr int N_SFB = BN / 128;                     // scale row tiles of B
  static constexpr int SFA_BYTES = (KS / KI) * SF_TILE;      // 2 KB
  static constexpr int SFB_BYTES = N_SFB * SFA_BYTES;
  static constexpr int STAGE = A_BYTES + B_BYTES + SFA_BYTES + SFB_BYTES;    // 38 KB (BN = 256), 28 KB (128)
  static constexpr int FIT = (227 * 1024 - CTL - 1024) / STAGE;
  static constexpr int STAGES = FIT > 7 ? 7 : FIT;
  static constexpr int SMEM = STAGES * STAGE + CTL + 1024;
  static constexpr int COL_ACC1 = BN == 256 ? 160 : 128;     // second accumulator
  static constexpr int OVERLAP = BN - COL_ACC1;              // columns it shares with the first (0: none)
  static constexpr int COL_SF = COL_ACC1 + BN;
  static constexpr int SF_COLS = 4 * (KS / KI) * (1 + N_SFB);                // one stage's scales: 48 or 32 columns
  static_assert(COL_SF + 2 * SF_COLS <= TMEM_COLS, "tensor memory budget");
  static_assert(BN % 64 == 0 && OVERLAP % 32 == 0, "the epilogue's pairs of chunks");
};
constexpr unsigned long long LIMIT_NS = 2000000000ull;

struct P4 {
  int M, N, K;
  int k_tiles;                               // 64-element tiles along the contraction (scale layout: padded)
  const float* sa; const float* sb;
  __nv_bfloat16* C; long long ldc;
  uint32_t* status;
  int one_by_one;                            // the producer's copies (see copies_one_by_one)
};

__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint32_t b, uint32_t n) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(b), "r"(n)); }
__device__ __forceinline__ void bar_expect(uint32_t b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t bar_try(uint32_t b, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.b32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(b), "r"(parity) : "memory");
  return ok;
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
struct Abort { volatile int* flag; uint32_t* status; };
__device__ __noinline__ bool bar_wait_slow(uint32_t b, uint32_t parity, const Abort& ab, uint32_t code) {
  const unsigned long long t0 = now_ns();
  for (uint32_t spin = 1;; ++spin) {
    if (bar_try(b, parity)) return true;
    if ((spin & 0xFF) == 0) {
      if (*ab.flag) return false;
      if (now_ns() - t0 > LIMIT_NS) { atomicCAS(ab.status, 0u, code); *ab.flag = 1; return false; }
    }
  }
}
__device__ __forceinline__ bool bar_wait(uint32_t b, uint32_t parity, const Abort& ab, uint32_t code) {
  return bar_try(b, parity) ? true : bar_wait_slow(b, parity, ab, code);
}
__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_leader(uint32_t addr) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void bar_arrive_cluster(uint32_t b) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(b) : "memory");
}
// Tiled TMA loads into this CTA's shared memory; the bytes are credited to `bar`, a barrier of the pair's leader.
__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void tma_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
               ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// When all tensor-core work issued so far has completed, arrive on the barrier at offset `bar` in both CTAs.
__device__ __forceinline__ void commit(uint32_t bar) {
  const uint16_t mask = 3;
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(mask) : "memory");
}
// Operand descriptor: rows of 128 bytes, 128-byte swizzle, contraction contiguous, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}
// Scale-tile descriptor for tcgen05.cp: 32 rows of 16 bytes, no swizzle, 8-row groups 128 B apart.
__device__ __forceinline__ uint64_t desc_sf(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 32) | ((uint64_t)1 << 46);
}
// Instruction descriptor of kind::mxf4nvf4: A = B = E2M1 (code 1), both K-major, E4M3 scales, N >> 3, M = 256 (the
// CTA pair) as M >> 4, K = 64.
__device__ __forceinline__ constexpr uint32_t idesc_fp4(int bn) {
  return (1u << 7) | (1u << 10) | ((uint32_t)(bn >> 3) << 17) | (0u << 23) | ((uint32_t)((2 * TM) >> 4) << 24);
}
__device__ __forceinline__ void cp_sf(uint32_t taddr, uint64_t sdesc) {
  asm volatile("tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}
__device__ __forceinline__ void mma_fp4(uint32_t d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t sfa, uint32_t sfb,
                                        uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %6, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::mxf4nvf4.block_scale.scale_vec::4X [%0], %1, %2, %3, [%4], [%5], p;\n\t}"
      ::"r"(d), "l"(da), "l"(db), "r"(idesc), "r"(sfa), "r"(sfb), "r"(acc) : "memory");
}
__device__ __forceinline__ void ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

template <int BN>
__global__ void __launch_bounds__(THREADS, 1)
nvfp4_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const __grid_constant__ CUtensorMap tmSA, const __grid_constant__ CUtensorMap tmSB, const P4 p) {
  using C4 = Cfg4<BN>;
  constexpr int STAGES = C4::STAGES;
  extern __shared__ uint8_t raw[];
  const uint32_t base = (s32(raw) + 1023u) & ~1023u;         // the same offset in both CTAs of the pair
  uint8_t* smem = raw + (base - s32(raw));
  const uint32_t ctl = base + STAGES * C4::STAGE;
  uint8_t* ctl_p = smem + STAGES * C4::STAGE;
  auto full = [&](int s) { return ctl + 8u * s; };
  auto empty = [&](int s) { return ctl + 8u * (STAGES + s); };
  auto tfull = [&](int a) { return ctl + 8u * (2 * STAGES + a); };
  auto tempty = [&](int a) { return ctl + 8u * (2 * STAGES + 2 + a); };      // leader only: accumulator drained by both CTAs
  const uint32_t shared_free = ctl + 8u * (2 * STAGES + 4);                  // leader only: a tile's shared columns drained
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(ctl_p + 8 * (2 * STAGES + 5));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(ctl_p + 8 * (2 * STAGES + 5) + 4);
  const Abort ab{abort_flag, p.status};
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cta_rank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  const int m_tiles = (p.M + 2 * TM - 1) / (2 * TM), n_tiles = (p.N + BN - 1) / BN;
  const int tiles = m_tiles * n_tiles;
  const int k_stages = (p.k_tiles + 3) / 4;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { bar_init(full(s), 1); bar_init(empty(s), 1); }
    for (int a = 0; a < 2; ++a) { bar_init(tfull(a), 1); bar_init(tempty(a), 2 * EPI_WARPS); }
    bar_init(shared_free, 2 * EPI_WARPS / 2);                // the four warps of the column half that holds them, per CTA
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(const_cast<uint32_t*>(tmem_slot))),
                 "r"((uint32_t)TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  fence_before();
  cluster_sync_all();
  fence_after();
  faar_pdl_sync();                                           // set-up done; now wait for the operands' kernels
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    auto load = [&](int mt, int nt, int ks, int stage) {
      const uint32_t sa = base + stage * C4::STAGE, sb = sa + C4::A_BYTES, sfa = sb + C4::B_BYTES, sfb = sfa + C4::SFA_BYTES;
      const uint32_t bar = map_to_leader(full(stage));
      if (rank == 0) bar_expect(full(stage), 2u * (uint32_t)C4::STAGE);
      tma_2d(sa, &tmA, ks * ROW_BYTES, mt * 2 * TM + (int)rank * TM, bar);
      tma_2d(sb, &tmB, ks * ROW_BYTES, nt * BN + (int)rank * (BN / 2), bar);
      tma_3d(sfa, &tmSA, 0, 4 * ks, 2 * mt + (int)rank, bar);
      tma_3d(sfb, &tmSB, 0, 4 * ks, nt * C4::N_SFB, bar);
    };
    int stage = 0; uint32_t phase = 0; bool ok = true;
    if (p.one_by_one && lane == 0) {                         // (see copies_one_by_one)
      for (int t = pair; t < tiles && ok; t += n_pairs) {
        const int mt = t % m_tiles, nt = t / m_tiles;
        for (int ks = 0; ks < k_stages; ++ks) {
          ok = bar_wait(empty(stage), phase ^ 1u, ab, 0x900u | stage);
          if (!ok) break;
          load(mt, nt, ks, stage);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
    // the whole warp, converged (see faar_elect_one): four copies a stage under `if (lane == 0)` took about 400 of the 512 clocks
    // that a stage's MMAs take, and a few stages' worth of a short contraction's whole time
    if (!p.one_by_one) {
      for (int t = pair; t < tiles && ok; t += n_pairs) {
        const int mt = t % m_tiles, nt = t / m_tiles;
        for (int ks = 0; ks < k_stages; ++ks) {
          ok = __all_sync(0xffffffffu, bar_wait(empty(stage), phase ^ 1u, ab, 0x900u | stage));
          if (!ok) break;
          if (faar_elect_one()) load(mt, nt, ks, stage);
          __syncwarp();
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
    if (!ok) { const unsigned long long t0 = now_ns(); while (now_ns() - t0 < 2000000ull) {} }
  } else if (warp == 1) {
    if (rank == 0) {                                         // the whole warp, converged (see faar_elect_one)
      int stage = 0; uint32_t phase = 0; int it = 0; bool ok = true;
      uint32_t sf = 0;                                       // which set of scale columns
      constexpr uint32_t idesc = idesc_fp4(BN);
      for (int t = pair; t < tiles && ok; t += n_pairs, ++it) {
        const int acc = it & 1;
        ok = bar_wait(tempty(acc), (uint32_t)((it >> 1) & 1) ^ 1u, ab, 0xA00u | acc);
        if (ok && C4::OVERLAP && it > 0) ok = bar_wait(shared_free, (uint32_t)((it - 1) & 1), ab, 0xA10u);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        fence_after();
        const uint32_t d = tmem + (uint32_t)(acc * C4::COL_ACC1);
        for (int ks = 0; ks < k_stages; ++ks) {
          ok = __all_sync(0xffffffffu, bar_wait(full(stage), phase, ab, 0xB00u | stage));
          if (!ok) break;
          fence_after();
          const int n_kt = min(4, p.k_tiles - 4 * ks);
          const uint32_t sa = base + stage * C4::STAGE, sb = sa + C4::A_BYTES, sfa = sb + C4::B_BYTES, sfb = sfa + C4::SFA_BYTES;
          const uint32_t ca = tmem + (uint32_t)C4::COL_SF + sf * (uint32_t)C4::SF_COLS, cb = ca + 16u;
          sf ^= 1u;
          const uint64_t da = desc_sw128(sa), db = desc_sw128(sb), dsa = desc_sf(sfa), dsb = desc_sf(sfb);
          if (faar_elect_one()) {
            auto issue = [&](int n) {
              // a B tile's scales for one MMA are N_SFB * 4 consecutive columns; in shared memory its row tiles are 2 KB apart
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                if (j < n) {
                  cp_sf(ca + 4u * j, dsa + (uint32_t)(j * (SF_TILE >> 4)));
#pragma unroll
                  for (int r = 0; r < C4::N_SFB; ++r)
                    cp_sf(cb + 4u * (uint32_t)(C4::N_SFB * j + r), dsb + (uint32_t)(r * (C4::SFA_BYTES >> 4) + j * (SF_TILE >> 4)));
                }
              }
#pragma unroll
              for (int j = 0; j < 4; ++j)            // 64 codes = 32 bytes further inside the swizzled row: +2
                if (j < n)
                  mma_fp4(d, da + 2u * j, db + 2u * j, idesc, ca + 4u * j, cb + 4u * (uint32_t)(C4::N_SFB * j), (ks | j) != 0 ? 1u : 0u);
            };
            if (n_kt == 4) issue(4); else issue(n_kt);
            commit(empty(stage));
          }
          __syncwarp();
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (ok && faar_elect_one()) commit(tfull(acc));
        __syncwarp();
      }
    }
  } else {
    const int quarter = warp & 3, half = (warp - 2) >> 2;    // lane quarter; column half of the tile
    const float alpha = *p.sa * *p.sb;
    int it = 0;
    for (int t = pair; t < tiles; t += n_pairs, ++it) {
      const int acc = it & 1;
      // whether a later tile waits for the shared columns, for this accumulator: else their release is not sent
      const bool next = t + n_pairs < tiles, again = t + 2 * n_pairs < tiles;
      bool ok = bar_wait(tfull(acc), (uint32_t)((it >> 1) & 1), ab, 0xC00u | acc);
      if (!__all_sync(0xffffffffu, ok)) break;
      fence_after();
      const int mt = t % m_tiles, nt = t / m_tiles;
      const int row = mt * 2 * TM + (int)rank * TM + quarter * 32 + lane;
      const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * C4::COL_ACC1);
      // the half whose columns the other accumulator shares starts at its shared end and reports when they are read
      const bool owner = C4::OVERLAP && half == (acc ^ 1);
      auto store = [&](int c, const uint32_t (&r)[16]) {
        const int col = nt * BN + c;
        if (row < p.M && col < p.N) {
          __nv_bfloat16* out = p.C + (long long)row * p.ldc + col;
          if (col + 16 <= p.N && ((reinterpret_cast<uintptr_t>(out) & 15) == 0)) {
            uint32_t o[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(r[2 * q]) * alpha, __uint_as_float(r[2 * q + 1]) * alpha);
              o[q] = *reinterpret_cast<uint32_t*>(&v);
            }
            if ((reinterpret_cast<uintptr_t>(out) & 31) == 0) {
              asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(out), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]),
                           "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]) : "memory");
            } else {
              reinterpret_cast<uint4*>(out)[0] = make_uint4(o[0], o[1], o[2], o[3]);
              reinterpret_cast<uint4*>(out)[1] = make_uint4(o[4], o[5], o[6], o[7]);
            }
          } else if (col + 16 <= p.N) {
            // a row off 16 bytes: values in pairs from the first 4-byte boundary on.  Single values -> pairs, rows of an odd number
            // of values, us: C[128, 16384] over 512 34.2 -> 13.8, [4096, 8192] over 2048 288 -> 103
            const bool odd = (reinterpret_cast<uintptr_t>(out) & 2) != 0;
            auto pair = [&](int q) {
              const __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(r[q]) * alpha, __uint_as_float(r[q + 1]) * alpha);
              return *reinterpret_cast<const uint32_t*>(&v);
            };
            if (odd) {
              out[0] = __float2bfloat16_rn(__uint_as_float(r[0]) * alpha);
#pragma unroll
              for (int q = 1; q < 15; q += 2) *reinterpret_cast<uint32_t*>(out + q) = pair(q);
              out[15] = __float2bfloat16_rn(__uint_as_float(r[15]) * alpha);
            } else {
#pragma unroll
              for (int q = 0; q < 16; q += 2) *reinterpret_cast<uint32_t*>(out + q) = pair(q);
            }
          } else {
#pragma unroll
            for (int q = 0; q < 16; ++q)
              if (col + q < p.N) out[q] = __float2bfloat16_rn(__uint_as_float(r[q]) * alpha);
          }
        }
      };
#pragma unroll 1
      for (int i = 0; i < BN / 32; i += 2) {                 // two loads, then both chunks' stores: 64 rows, 28672 x 256 7.0 -> 6.3 us
        const int c0 = half == 0 ? 16 * i : BN - 16 - 16 * i, c1 = half == 0 ? c0 + 16 : c0 - 16;
        uint32_t r0[16], r1[16];
        ld16(trow + (uint32_t)c0, r0);
        ld16(trow + (uint32_t)c1, r1);
        if (owner && i == C4::OVERLAP / 16 - 2) {
          fence_before();
          __syncwarp();
          if (next && lane == 0) bar_arrive_cluster(map_to_leader(shared_free));
        }
        store(c0, r0);
        store(c1, r1);
        __syncwarp();                                        // the next load of tensor memory wants the whole warp
      }
      fence_before();
      __syncwarp();
      if (again && lane == 0) bar_arrive_cluster(map_to_leader(tempty(acc)));
    }
  }
  __syncwarp();
  // Neither CTA leaves while the other can still use its memory or arrive on its barriers; all of that has been waited for
  // by now, so a relaxed arrival does, which does not wait for this CTA's results to reach L2.  After a wait that gave up
  // it may still be on its way: then the full form, and some time.
  fence_before();
  __syncthreads();
  if (*abort_flag) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  else asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (*abort_flag) { const unsigned long long t0 = now_ns(); while (now_ns() - t0 < 2000000ull) {} }
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)TMEM_COLS) : "memory");
  }
}

typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// rows x (K/2) bytes, bytes of a row contiguous; box = 128 bytes x box_rows.
int byte_map(faar_ctx* ctx, CUtensorMap* map, const void* ptr, int rows, int K, int box_rows) {
  cuuint64_t dims[2] = {(cuuint64_t)(K / 2), (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(K / 2)};
  cuuint32_t box[2] = {(cuuint32_t)ROW_BYTES, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  CUresult r = reinterpret_cast<EncodeFn>(ctx->encode_tiled)(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(ptr), dims,
                                                             strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                                             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : (int)cudaErrorInvalidValue;
}
// Tiled scales: [row tile][k tile][128 words]; box = four k tiles of box_rows row tiles.
int scale_map(faar_ctx* ctx, CUtensorMap* map, const void* ptr, int row_tiles, int k_tiles, int box_rows) {
  cuuint64_t dims[3] = {(cuuint64_t)(SF_TILE / 4), (cuuint64_t)k_tiles, (cuuint64_t)row_tiles};
  cuuint64_t strides[2] = {(cuuint64_t)SF_TILE, (cuuint64_t)SF_TILE * (cuuint64_t)k_tiles};
  cuuint32_t box[3] = {(cuuint32_t)(SF_TILE / 4), (cuuint32_t)(KS / KI), (cuuint32_t)box_rows};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = reinterpret_cast<EncodeFn>(ctx->encode_tiled)(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<void*>(ptr), dims,
                                                             strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                                             CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : (int)cudaErrorInvalidValue;
}

// 256-wide tiles move the fewest operand bytes per flop; 128-wide ones are taken while 256-wide tiles would not give
// every CTA pair one (a token batch of up to 256 rows, a small layer), where spreading the weights over twice as many
// SMs counts for more.
bool pick_wide4(int M, int N, int pairs) {
  return (long long)((M + 2 * TM - 1) / (2 * TM)) * ((N + 255) / 256) >= pairs;
}

// Where one lane issues the producer's copies one by one, about 0.2 us a stage, instead of an elected lane of the converged warp
// all at once, which is 3 to 13 % faster in general.  Up to three stages a tile: there is nothing to get ahead of (200 products of up to 300 rows,
// at once 1.0 to 1.5 % slower, 4.9 % at most).  And with fewer than 128 rows of A and less than 128 KB of them in all, where pairs that
// ask for a whole ring at a time hold one another up once more pairs are at work (in the last wave) than one die has, with up to 8 rows,
// depending on the addresses, from a third of the pairs on (1 to 8 rows, 25 to 37 tiles, 0.90 to 1.12, on average 1.01 times as long).
// One by one / at once, us: 8 rows, 8192 x 2048 5.8 / 6.3, x 8192 13.1 / 16.0, 16384 x 8192 23.0 / 31.4; 64 rows, 8192 x 2048 5.8 / 6.3,
// x 4096 (128 KB) 8.1 / 7.5; 127 rows, 8192 x 2048 6.45 / 6.86, 128 rows 6.4 / 6.1; 1 row, 4096 x 2048 5.9 / 6.5, 64 rows 5.7 / 5.4,
// 11008 x 2048 (86 tiles, 12 in the last wave) 8.2 / 7.7.
bool copies_one_by_one(int M, int K, int bn, long long tiles, int pairs) {
  if (K <= 3 * KS) return true;
  return bn == 128 && M < TM && (long long)M * K < 2 * 131072 && (tiles - 1) % pairs >= (M <= 8 ? pairs / 3 : pairs / 2);
}

template <int BN>
int launch4(faar_ctx* ctx, const uint8_t* A, const uint8_t* sfa, const uint8_t* B, const uint8_t* sfb, P4& p) {
  using C4 = Cfg4<BN>;
  auto kern = nvfp4_gemm_kernel<BN>;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.blockDim = dim3(THREADS, 1, 1);
  cfg.dynamicSmemBytes = C4::SMEM;
  cfg.stream = ctx->stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  int e = faar_allow_smem(ctx, (const void*)kern, C4::SMEM);
  if (e) return e;
  const int max_pairs = faar_max_clusters(ctx, FAAR_GEMM_VARIANTS + (BN == 256), 0, (const void*)kern, &cfg);
  CUtensorMap tmA, tmB, tmSA, tmSB;
  e = byte_map(ctx, &tmA, A, p.M, p.K, TM);
  if (!e) e = byte_map(ctx, &tmB, B, p.N, p.K, BN / 2);
  if (!e) e = scale_map(ctx, &tmSA, sfa, (p.M + 127) / 128, p.k_tiles, 1);
  if (!e) e = scale_map(ctx, &tmSB, sfb, (p.N + 127) / 128, p.k_tiles, C4::N_SFB);
  if (e) return e;
  const long long tiles = (long long)((p.M + 2 * TM - 1) / (2 * TM)) * ((p.N + BN - 1) / BN);
  p.one_by_one = copies_one_by_one(p.M, p.K, BN, tiles, ctx->num_sms / 2);
  cfg.gridDim = dim3(2 * (unsigned)(tiles < max_pairs ? tiles : max_pairs), 1, 1);
  faar_prof_scope ps(ctx, FAAR_K_NVFP4_GEMM);
  cudaError_t ce = cudaLaunchKernelEx(&cfg, kern, tmA, tmB, tmSA, tmSB, p);
  if (ce != cudaSuccess) return (int)ce;
  return (int)cudaGetLastError();
}

}  // namespace

int faar_launch_nvfp4_gemm(faar_ctx* ctx, int M, int N, int K, const uint8_t* A, const uint8_t* sfa, const float* sa,
                           const uint8_t* B, const uint8_t* sfb, const float* sb, void* C, int64_t ldc, uint32_t* status) {
  P4 p;
  p.M = M; p.N = N; p.K = K; p.k_tiles = (K + KI - 1) / KI;
  p.sa = sa; p.sb = sb; p.C = reinterpret_cast<__nv_bfloat16*>(C); p.ldc = ldc; p.status = status;
  return pick_wide4(M, N, ctx->num_sms / 2) ? launch4<256>(ctx, A, sfa, B, sfb, p) : launch4<128>(ctx, A, sfa, B, sfb, p);
}
