// Internal declarations shared by the translation units of libfaar.so.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "faar.h"

#include <vector>

constexpr int FAAR_GEMM_VARIANTS = 8;     // REF, FWD, BWD x 4 optimiser / chaining variants
constexpr int FAAR_PAIR_KERNELS = FAAR_GEMM_VARIANTS + 2;   // and the NVFP4 GEMM's 128- and 256-wide tiles

constexpr int FAAR_SPLIT_PLANS = 16;
struct faar_split_plan { int mode, m_tiles, n_main, narrow, bn, full; };   // GEMM tail split of a tile grid, as chosen

struct faar_ctx {
  int device;
  int num_sms;
  cudaStream_t stream;
  int last_cuda_error;
  void* encode_tiled;  // cuTensorMapEncodeTiled, resolved through the runtime
  int tune_bn;                            // 0 = choose the GEMM tile width automatically
  int tune_tail;                          // -1 = choose the tail split automatically, else columns to split
  int tune_wide;                          // 256 x 512 GEMM tiles: 1 = wherever the shape allows, 0 = never, -1 (default) = pick_wide's rule; 0 and 1 keep contractions whole
  int tune_attention_fragments;           // attention: 0 = tcgen05 kernels, 2 = mma.sync kernels (head_dim 64), 1 = the shared-memory fragment kernels
  int last_gemm_bn, last_gemm_pairs, last_gemm_split;   // what the last GEMM launch used
  std::vector<const void*> smem_set;      // kernels whose dynamic shared-memory limit has been raised on this device
  faar_split_plan split_plans[FAAR_SPLIT_PLANS];          // the last ones used
  unsigned next_plan;
  // chained steps: the workspace and the beta of the forward operand that the last backward call wrote
  const void* wsoft_ws;
  float wsoft_beta;
  // host-batch path (faar_layer_step_host): copies run on their own stream, ordered by events
  cudaStream_t copy_stream;
  cudaEvent_t ev_copied, ev_done[2];
  unsigned long long host_calls;
  const void* last_staging;
  // faar_model_forward_both: the frozen pass runs on its own stream
  cudaStream_t side_stream;
  cudaEvent_t ev_fork, ev_join;
  // per-kernel timing (faar_profile_begin / faar_profile_end)
  bool prof_on;
  int prof_used;                          // event pairs used since faar_profile_begin
  std::vector<cudaEvent_t> prof_events;   // 2 per launch: start, stop
  std::vector<int> prof_kernel;           // kernel id per pair
};

// Brackets one kernel launch with a pair of CUDA events when profiling is on.
struct faar_prof_scope {
  faar_ctx* c;
  int pair;
  faar_prof_scope(faar_ctx* ctx, int kernel_id);
  ~faar_prof_scope();
};

// Raises a kernel's dynamic shared-memory limit, once per context (the call costs about as much host time as a launch's
// argument checks and every launch of a small layer would pay it).  The context's device is current.
// carveout: the part of the SM's memory that is preferred as shared memory, in percent; -1 leaves it to the driver.
int faar_allow_smem(faar_ctx* c, const void* kernel, int bytes, int carveout = -1);
// How many clusters of `kernel` (launched as *cfg, which says their size 2 << size; its grid ignored) the context's device
// holds at once: a fact of device and kernel (a GPC with an odd SM count strands one SM), asked once per device and process.
constexpr int FAAR_CLUSTER_SIZES = 3;     // 2, 4, 8 CTAs
int faar_max_clusters(faar_ctx* c, int slot, int size, const void* kernel, cudaLaunchConfig_t* cfg);
// The number from the query's answer; `most` is what the SM count allows.  Without an answer every SM is counted for pairs,
// which every launch needs, and no larger cluster: a contraction is then not split over one that the device may refuse.
inline int faar_cluster_count(bool answered, int n, int size, int most) {
  if (!answered || n <= 0) return size ? 0 : most;
  return n < most ? n : most;
}

// Launch with stream serialisation relaxed (programmatic dependent launch): the kernel's CTAs may be scheduled while the
// kernel before it drains; the kernel itself waits (faar_pdl_sync) before it touches global memory.
template <typename... KArgs, typename... Args>
static inline cudaError_t faar_launch_pdl(faar_ctx* ctx, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = ctx->stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ---- workspace layout -------------------------------------------------------
// [0, 256)            header: word 0 = status (0 = ok), bytes 8..15 = the final sums of a
//                     dW launch while its CTAs finish (zero between launches), bytes 16..23 = tensor maximum of
//                     the last set-up pass (high word: the pass's serial number, low word: max |W| bits),
//                     bytes 24..27 = clusters of an alignment-loss launch that have finished (zero between launches),
//                     bytes 64..127 = a bit per CTA of a dW launch whose Round Loss sum lies in the Round region
//                     (zero between launches)
// [256, 256+P)        loss partials (float): MSE region then Round region
// [..]                W_soft bf16 [O,K]
// [..]                dYt bf16 [O, ceil8(T)]
constexpr size_t FAAR_WS_HEADER = 256;
constexpr int FAAR_MAX_PARTIALS = 16384;  // per loss term

struct faar_ws_layout {
  size_t off_mse_partials, off_round_partials, off_wsoft, off_dyt, total;
  int64_t ld_dyt;
};

static inline size_t faar_align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static inline faar_ws_layout faar_ws_plan(const faar_shape* s) {
  faar_ws_layout l;
  l.ld_dyt = ((int64_t)s->T + 7) / 8 * 8;
  size_t off = FAAR_WS_HEADER;
  l.off_mse_partials = off;
  off += sizeof(float) * FAAR_MAX_PARTIALS;
  l.off_round_partials = off;
  off += sizeof(float) * FAAR_MAX_PARTIALS;
  off = faar_align_up(off, 1024);
  l.off_wsoft = off;
  off += (size_t)s->O * (size_t)s->K * 2;
  off = faar_align_up(off, 1024);
  l.off_dyt = off;
  off += (size_t)s->O * (size_t)l.ld_dyt * 2;
  l.total = faar_align_up(off, 1024);
  return l;
}

// The per-weight state a dW product updates: one linear, or (row-major operands) up to three whose output rows are
// stacked, each with its own tensors and Round Loss weight.
constexpr int FAAR_MAX_SEGMENTS = 3;
struct faar_bwd_state {
  float* V; const uint8_t* code; const uint8_t* scales; const float* s_global;
  float* adam_m; float* adam_u; float* dV;
  float lam_over_n;
  int rows;               // output rows of this linear (a multiple of 8 where several are stacked)
};

// ---- launchers (each returns a cudaError_t as int) ---------------------------
int faar_launch_softquant_init(faar_ctx*, const faar_shape*, const void* W, float s_global_in,
                               uint8_t* scales, float* s_global_out, uint8_t* code, float* V,
                               unsigned long long* amax_word);
int faar_launch_nvfp4_expand(faar_ctx*, int rows, int K, const uint8_t* packed, const uint8_t* scales, void* out, int64_t ld);
// head_dim D = 64 or 128 on the tcgen05 tensor cores
int faar_launch_attention_fwd_tc(faar_ctx*, int B, int S, int H, int Hkv, int D, const void* q, int64_t ldq, const void* k,
                                 const void* v, int64_t ldk, void* out, int64_t ldo, float* lse, float scale_log2);
// rope: dq and dk turn back by their row's angles, [D / 2, B S] sines and cosines, on the way out (null: they don't)
int faar_launch_attention_bwd_tc(faar_ctx*, int B, int S, int H, int Hkv, int D, const void* q, int64_t ldq, const void* k,
                                 const void* v, int64_t ldk, const void* dout, int64_t ldo, const float* lse,
                                 const float* dsum, int sum_parts, void* dq, void* dk, void* dv, float scale_log2, const float2* rope);
int faar_attention_tc_status(uint32_t* code_out);
int faar_launch_softquant_eval(faar_ctx*, const faar_shape*, const float* V, const uint8_t* code,
                               const uint8_t* scales, const float* s_global, float beta,
                               float* W_soft, float* h, __nv_bfloat16* W_soft_bf16,
                               float* W_operand_f32 = nullptr);
// BF16 soft weights of several linears (1 .. FAAR_MAX_SOFT_ITEMS), `weights` (a multiple of 16, below 2^40) each
constexpr int FAAR_MAX_SOFT_ITEMS = 28;
struct faar_soft_item { const float* V; const uint8_t* code; const uint8_t* scales; const float* s_global; __nv_bfloat16* out; int64_t weights; };
int faar_launch_soft_weights(faar_ctx*, int n, const faar_soft_item* item, float beta);
int faar_launch_act_fakequant(faar_ctx*, int T, int K, const void* X, int64_t ldx, float s_global_in, void* Xq,
                              int64_t ldq, float* s_global_out, uint8_t* packed, uint8_t* scales,
                              unsigned long long* amax_word);
int faar_launch_transpose_bf16(faar_ctx*, int rows, int cols, const void* in, int64_t ld_in, void* out,
                               int64_t ld_out);
int faar_launch_swizzle_scales(faar_ctx*, int rows, int cols, const uint8_t* in, uint8_t* out);
// Eq. 6's data terms: one partial of each per CTA or cluster, at most one per token; `finished` is zero between launches
int faar_launch_align_loss(faar_ctx*, int T, int vocab, int hidden, const void* Z_fp, const void* Z_q, int64_t ldz,
                           const void* H_fp, const void* H_q, int64_t ldh, float tau, float lambda_kl, void* dZ_q,
                           void* dH_q, float* kl_partials, float* mse_partials, uint32_t* finished, float* loss_out2,
                           const float2* stats_fp = nullptr, const float2* stats_q = nullptr);      // of the logits' products, both or none
// The statistics that a product of these logits leaves, [T, ceil(vocab / 128)]
int faar_launch_logit_stats(faar_ctx*, int T, int vocab, const void* Z, int64_t ldz, float tau, float2* stats);
int faar_launch_silu_mul(faar_ctx*, int rows, int cols, const void* gate, int64_t ldg, const void* up, int64_t ldu,
                         void* out, int64_t ldo);
int faar_launch_rmsnorm(faar_ctx*, int rows, int cols, const void* x, int64_t ldx, const void* b, int64_t ldb,
                        void* sum_out, int64_t lds, const float* g, float eps, void* y, int64_t ldy, float* rstd);
int faar_launch_rmsnorm_bwd(faar_ctx*, int rows, int cols, const void* dy, const void* dy2, const void* dy3, int64_t lddy,
                            const void* x, int64_t ldx, const float* g, const float* rstd, const void* add, int64_t ldadd,
                            void* dx, int64_t lddx);
int faar_launch_rope(faar_ctx*, int rows, int n_heads, int head_dim, const void* x, int64_t ldx, const int* pos, float theta,
                     int inverse, void* y, int64_t ldy);
int faar_launch_silu_mul_bwd(faar_ctx*, int rows, int cols, const void* dout, int64_t ldd, const void* gate, int64_t ldg,
                             const void* up, int64_t ldu, void* dgate, int64_t lddg, void* dup, int64_t lddu);
int faar_launch_embedding(faar_ctx*, int rows, int cols, int vocab, const void* table, int64_t ldt, const int* tokens,
                          void* out, int64_t ldo);
// How a model's pass begins: x = the tokens' rows of the table, y = rmsnorm(x), and every row's rotary angles, [head_dim / 2,
// rows] sines and cosines
int faar_launch_embed_rmsnorm(faar_ctx*, int rows, int cols, int vocab, const void* table, const int* tokens, void* x, const float* g,
                              float eps, void* y, float* rstd, const int* pos, int head_dim, float theta, float2* rope);
int faar_launch_add(faar_ctx*, int rows, int cols, const void* a, int64_t lda, const void* b, int64_t ldb, void* out,
                    int64_t ldo);
int faar_launch_attention_fwd(faar_ctx*, int B, int S, int H, int Hkv, int D, const void* q, int64_t ldq, const void* k,
                              const void* v, int64_t ldk, void* out, int64_t ldo, float* lse);
int faar_launch_attention_bwd(faar_ctx*, int B, int S, int H, int Hkv, int D, const void* q, int64_t ldq, const void* k,
                              const void* v, int64_t ldk, const void* out, const void* dout, int64_t ldo, const float* lse,
                              float* dsum, void* dq, void* dk, void* dv, const float2* rope = nullptr, int sum_parts = 0);
int faar_launch_nvfp4_gemm(faar_ctx*, int M, int N, int K, const uint8_t* A, const uint8_t* sfa, const float* sa,
                           const uint8_t* B, const uint8_t* sfb, const float* sb, void* C, int64_t ldc, uint32_t* status);
int faar_launch_round_partials(faar_ctx*, const float* V, int64_t N, float* partials, int* n_partials);
// out[0] = scale0 * sum(p0[0..n0)), out[1] = scale1 * sum(p1[0..n1)) (either may have n = 0 -> skipped)
int faar_launch_finalize(faar_ctx*, const float* p0, int n0, float scale0, float* out0, const float* p1,
                         int n1, float scale1, float* out1);
int faar_launch_harden_pack(faar_ctx*, const faar_shape*, const float* V, const uint8_t* code,
                            const uint8_t* scales, const float* s_global, uint8_t* packed,
                            uint8_t* scales_out, uint8_t* decisions, void* W_final, int wfinal_dtype);

// dW products with chain rule and update on row-major operands dY [T, ldy], X [T, ldx]; the segments' rows stacked in dY's
// columns.  hp has been checked.
// beside: it runs next to the launches before it (see faar_gemm_args)
int faar_bwd_group(faar_ctx*, int n_seg, faar_bwd_state* seg, int T, int K, const faar_hparams* hp, const void* dY, int64_t ldy,
                   const void* X, int64_t ldx, void* workspace, bool beside = false);
int faar_check_hparams(const faar_hparams* hp, bool need_opt);

enum { FAAR_GATED_FWD = 1, FAAR_GATED_BWD = 2 };
enum { FAAR_GEMM_REF = 0, FAAR_GEMM_FWD = 1, FAAR_GEMM_BWD = 2 };

struct faar_gemm_args {
  int mode;
  int M, N, Kc;           // C[M,N] = A[M,Kc] * B[N,Kc]^T, both operands bf16 with Kc contiguous (REF: the launch may exchange them)
  const void* A; int64_t lda;
  const void* B; int64_t ldb;
  int beside;             // BWD: 1: starts next to the launches before it, back to the last one that waits first (faar_pdl_wait_first).  Its
                          // inputs must be complete when that one's wait is, nothing since may write what it reads or read what it
                          // writes, and each launch since must join its predecessor before it ends: a plain product or dK / dV first, then
                          // dQ and dW products in any number
  int ahead;              // FWD, BWD: 1: of what the launch before it on the stream writes it needs the A operand alone, and that launch lets
                          // it start once all before is complete (faar_pdl_wait_first)
  int whole;              // 1: the contraction is not split over CTA pairs (the order of its sums is that of one pair)
  int a_mn, b_mn;         // 1: the operand is stored with M (N) contiguous instead: A[Kc, M] (lda), B[Kc, N] (ldb)
  uint32_t* status;       // workspace status word
  // REF / FWD
  void* Yout; int yout_dtype; int64_t ldy;     // REF: [M, ldy]; FWD: [N(T), M(O)] written transposed, nullable
  const void* Yref; int yref_dtype;            // FWD
  int yref_t;                                  // FWD: Y stored transposed [O, ldy]; REF: rows of Yout padded to 16 columns
  int gated;                                   // REF: an epilogue of the gated product, FAAR_GATED_FWD or FAAR_GATED_BWD (0: plain)
  void* act; const void* gate_up;              // and its further tensors (see faar_gemm.cu)
  float2* stats; float stats_c;                // REF: softmax statistics of every row, [M, ceil(N / 128)] (null: not wanted)
  const void* sum_with; float* sums;           // REF: sums of the result times sum_with [M, ldy] over the sum_dim columns of each head, as
  int sum_dim; int* sum_parts;                 // sum_parts parts (set by the launch) [parts, heads, M] (sums null: not wanted)
  const float2* rope;                          // REF: the first rope_cols columns of the result are heads that turn by their row's
  int rope_cols, head_dim;                     // angles, [head_dim / 2, M] sines and cosines (null: none do)
  __nv_bfloat16* dYt; int64_t ld_dyt;          // FWD: [M(O), ld_dyt]
  float mse2c;                                 // FWD: 2 * mse_scale
  float act_scale;                             // FWD, BWD: tensor scale of quantised activations (1 = none)
  float* partials;                             // FWD: sum r^2 partials
  // BWD: M = O, N = K
  int n_seg; faar_bwd_state seg[FAAR_MAX_SEGMENTS];
  float beta, lr, b1, b2, eps, inv_bc1, inv_bc2; int opt;
  // BWD, optional: also write the next step's BF16 operand W_soft(V', beta_next) (null = not wanted)
  __nv_bfloat16* wsoft_next; float beta_next;
  // BWD, optional: final loss sums by the last CTA (fin_out2 null = not wanted)
  unsigned long long* fin_word; unsigned long long* fin_far; double* fin_far_sums; const float* fin_mse_partials; int fin_n_mse; float fin_scale_mse, fin_scale_round;
  float* fin_out2;
};
// n_partials_out: number of floats a FWD launch writes to args.partials
int faar_launch_gemm(faar_ctx*, const faar_gemm_args*, int* n_partials_out);
bool faar_logit_stats_fit(const faar_ctx*, int T, int vocab);
bool faar_logit_stats_pays(const faar_ctx*, int T, int vocab);
int faar_check_logit_stats(faar_ctx*, int T, int vocab, const void* stats, size_t stats_bytes);      // a caller's buffer of them
int faar_gemm_max_partials(const faar_ctx*, int M, int N);
int faar_launch_wait_selftest(faar_ctx*, uint32_t* status, unsigned long long limit_ns);

// ---- device helpers -----------------------------------------------------------
#ifdef __CUDACC__

// E2M1 magnitude of code c (0..7): 0, .5, 1, 1.5, 2, 3, 4, 6.
__device__ __forceinline__ float faar_node(int c) {
  int e = c >> 1, m = c & 1;
  // e == 0: m * 0.5 ; else (1 + m/2) * 2^(e-1)
  float normal = __uint_as_float(((uint32_t)(e + 126) << 23) | ((uint32_t)m << 22));
  return e == 0 ? 0.5f * (float)m : normal;
}

// width of interval k (0..6): .5 .5 .5 .5 1 1 2
__device__ __forceinline__ float faar_width(int k) { return k < 4 ? 0.5f : (k < 6 ? 1.0f : 2.0f); }

// FP8 E4M3 byte -> float (finite codes only).
__device__ __forceinline__ float faar_e4m3_to_float(uint32_t b) {
  uint32_t h;                                   // exact: E4M3 is a subset of F16
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h) : "h"((uint16_t)(b & 0x7Fu)));
  return __low2float(*reinterpret_cast<const __half2*>(&h));
}

// Non-negative float -> nearest finite E4M3 byte, ties to even, saturating at 448 (also from infinity and NaN).
__device__ __forceinline__ uint32_t faar_float_to_e4m3(float q) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(0.f), "f"(fminf(q, 448.0f)));
  return r;
}

// Eq. 3 in FP32 with a relative error of a few 1e-7 over the whole range of h, also where h is tiny.
// z = beta*(v-0.5) is kept as an unevaluated sum (v-0.5 is exact or off by < 2^-26; the product's
// rounding error is recovered with one FMA), -|z|*log2(e) likewise, so the argument of the hardware
// 2^x carries no error that grows with |z|; the low parts enter as a first-order correction.
__device__ __forceinline__ float faar_sigmoid_precise(float beta, float v) {
  const float d = __fsub_rn(v, 0.5f);
  const float zh = __fmul_rn(beta, d);
  const float zl = __fmaf_rn(beta, d, -zh);              // exact error of the product
  const float az = -fabsf(zh);
  const float sl = zh >= 0.f ? -zl : zl;                  // low part of -|z| (sign follows zh)
  const float L1 = 1.4426950216293335f;                   // float(log2 e)
  const float L2 = 1.9259629911266175e-8f;                // log2 e - L1
  const float th = __fmul_rn(az, L1);
  float tl = __fmaf_rn(az, L1, -th);
  tl = __fmaf_rn(az, L2, tl);
  tl = __fmaf_rn(sl, L1, tl);
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(th));
  e = __fmaf_rn(e, tl * 0.6931471805599453f, e);          // 2^(th+tl) = 2^th (1 + tl ln 2)
  const float hs = __fdividef(1.0f, 1.0f + e);            // sigmoid(|z|)
  return zh >= 0.f ? hs : __fmul_rn(e, hs);               // sigmoid(-|z|) = e / (1 + e)
}

// Eq. 3 as the forward GEMM's BF16 operand is built (relative error below 3e-6):
// h = 1 / (1 + 2^(-z log2 e)), z = beta (v - 0.5), with beta log2(e) rounded once, the exponent formed
// in one FMA, hardware 2^x and reciprocal.  A 2^x that overflows (z < -88) gives h = 0, the value's
// rounding.  nbl = -(beta * log2 e), hbl = -nbl / 2 (faar_operand_consts).
__device__ __forceinline__ void faar_operand_consts(float beta, float* nbl, float* hbl) {
  *nbl = -__fmul_rn(beta, 1.4426950408889634f);
  *hbl = -0.5f * *nbl;
}
__device__ __forceinline__ float faar_sigmoid_operand(float nbl, float hbl, float v) {
  float e, h;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(fmaf(nbl, v, hbl)));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(h) : "f"(1.0f + e));
  return h;
}
// The operand value before its rounding to BF16: (lo + h * width) * s with the sign of w, in exactly
// these operations wherever it is produced (soft-weights kernel, dW epilogue), so that both give the
// same bits.  lo and width may carry the sign already (rounding is symmetric).
__device__ __forceinline__ float faar_operand_weight(float h, float lo, float width, float s) {
  return fmaf(h, width, lo) * s;
}

// Eq. 2 in FP32: sign * (lo + h * (hi - lo)) * s for the nibble (sign<<3 | k).
__device__ __forceinline__ float faar_soft_weight(float h, uint32_t nib, float s) {
  int k = nib & 7;
  float mag = __fmul_rn(__fmaf_rn(h, faar_width(k), faar_node(k)), s);
  return (nib & 8) ? -mag : mag;
}

// Programmatic dependent launch: the step's kernels are launched with stream serialisation relaxed, so
// that a kernel's CTAs may start (and run their set-up) on SMs that the previous kernel has already
// left.  faar_pdl_sync() lets the next kernel do the same and then waits until the previous kernel has
// completed and its memory is visible; nothing before it may touch global data.
__device__ __forceinline__ void faar_pdl_sync() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The other order, for a kernel that the next one may run next to (an input gradient and the dW product of the same dY): once
// every CTA is past its wait, all that came before is complete, so a dependent that needs nothing of THIS kernel starts at
// once, on the SMs that are free or become so, and only has to wait (faar_pdl_join) before it ends: what follows it then
// finds both complete.  Several may follow one another like this.  The dW products of a backward pass next to the input
// gradients and dQ next to dK / dV, alignment step, us: four 128-wide blocks on 1200 tokens 531 -> 459, two of 512 on 400 357 -> 318,
// two of 2048 / 8192 on 700 1832 -> 1803, two of 2048 / 6144 on 500 1350 -> 1323; with two dW products next to gate / up's input
// gradient, and the output projection's next to dQ, 436 -> 403, 306 -> 283, 1775 -> 1770 and 1303 -> 1291.
__device__ __forceinline__ void faar_pdl_wait_first() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void faar_pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void faar_pdl_join() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// One lane of a converged warp.  A warp that issues tensor-core instructions runs its loop with all lanes and guards
// only those instructions with this, so that the descriptors stay in uniform registers; under `if (lane == 0)` every
// operand is moved there first, about 65 clocks per instruction, and the issuing thread becomes the bottleneck
// (NVFP4 GEMM, C[4096, 2048], K = 8192: 71 us against 33.8 us).  The same for a warp that issues copies: two or four a stage and
// their barrier took most of what a stage of a narrow tile lasts.  Step of 64 x 8192 at 300 tokens 44.6 -> 42.6 us, 512 x 2048 at 4096 30.2
// -> 29.3, 512 x 512 at 512 16.9 -> 16.1, 128 x 256 at 1024 12.8 -> 12.5; alignment step of two 512-wide blocks on 400 tokens 270.6 ->
// 262.6; NVFP4 product of 8 tokens, 2048 x 8192, with its quantiser 18.5 -> 16.5, of 1000 tokens, 2048 x 4096, 9.1 -> 8.4.
__device__ __forceinline__ bool faar_elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

// sigmoid(x) in FP32: 1 / (1 + e^-x) with the library exponential (relative error ~1e-7) and the hardware
// reciprocal (rcp.approx: relative error below 2^-22); e^-x overflowing to +inf gives 0, the limit.
__device__ __forceinline__ float faar_sigmoid(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + expf(-x)));
  return r;
}
// The gated product silu(g) u and its backward: with s = sigmoid(g),  dg = d u s (1 + g (1 - s)),  du = d g s.
__device__ __forceinline__ float faar_silu_mul(float g, float u) { return g * faar_sigmoid(g) * u; }
__device__ __forceinline__ void faar_silu_mul_bwd(float d, float g, float u, float& dg, float& du) {
  const float s = faar_sigmoid(g);
  dg = d * u * s * fmaf(g, 1.0f - s, 1.0f);
  du = d * g * s;
}

// Rotary position embedding, half-split pairing: element i (i < head_dim / 2) of a head and element i + head_dim / 2 turn by
// pos theta^(-2 i / head_dim); the backward pass of an orthogonal map is the rotation by the negative angle.
__device__ __forceinline__ float faar_rope_frequency(int i, int head_dim, float log2_theta) {
  return exp2f(-2.0f * (float)i / (float)head_dim * log2_theta);
}
__device__ __forceinline__ void faar_rope_turn(float& a, float& b, float sn, float cs) {
  const float x = fmaf(a, cs, -(b * sn)), y = fmaf(b, cs, a * sn);
  a = x;
  b = y;
}

__device__ __forceinline__ float faar_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Maximum m of c z and sum s of 2^(c z - m) over a row's values z so far, 16 more of them taken in; before the first, m = -inf, s = 0.
// One order of every sum wherever a row's statistics are formed: 128 columns in turn.
__device__ __forceinline__ void faar_stats_update(const float (&z)[16], float c, float& m, float& s) {
  float mx = -INFINITY;
#pragma unroll
  for (int j = 0; j < 16; j += 2) mx = fmaxf(mx, fmaxf(z[j], z[j + 1]));
  mx *= c;                                            // c > 0: scaling keeps the order
  if (mx > m) { s *= faar_ex2(m - mx); m = mx; }      // 2^-inf = 0 on the first 16
#pragma unroll
  for (int j = 0; j < 16; ++j) s += faar_ex2(fmaf(z[j], c, -m));
}

__device__ __forceinline__ float faar_warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

#endif  // __CUDACC__
