// Forward and backward passes of a whole decoder model (full-model alignment, Procedure steps 16-17 and 21-23): the
// sequence of kernel launches for every block, enqueued by one call.  No arithmetic here and no kernels of its own.
//
// Why native: a step is a chain of 27 launches per block (7 in each forward pass, 12 in the backward pass, soft weights), many
// of a few microseconds each.  Issued one by one from Python a launch cost 7.5 us of host time, more than the kernels of a small
// model take: an alignment step of two 128-wide blocks on 192 tokens took 770 us for 500 us of device time (177 us as it is
// now).  Activations live in one caller-owned arena per pass at offsets that depend on the sizes alone.
#include <math.h>

#include "faar_internal.cuh"

namespace {

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

struct Sizes {
  size_t T;
  int d, qd, kvd, qkv, f, H, hd;
  size_t seq_rows;                            // floats of one lse array
};
Sizes sizes(const faar_model* m, int batch, int seq) {
  Sizes s;
  s.T = (size_t)batch * seq;
  s.d = m->hidden; s.qd = m->n_heads * m->head_dim; s.kvd = m->n_kv_heads * m->head_dim; s.qkv = s.qd + 2 * s.kvd; s.f = m->ffn;
  s.H = m->n_heads; s.hd = m->head_dim;
  s.seq_rows = s.T * m->n_heads;
  return s;
}

// Byte offsets of a block's saved activations inside its part of the arena.
struct BlockLayout {
  size_t x_in, hn, rstd1, qkv, a, lse, x_mid, rstd2, mn, gu, act, bytes;
  BlockLayout(const Sizes& s, bool keep) {
    size_t o = 0;
    auto take = [&](size_t n) { const size_t at = o; o += align256(n); return at; };
    x_in = take(s.T * s.d * 2); hn = take(s.T * s.d * 2); rstd1 = take(s.T * 4);
    qkv = take(s.T * s.qkv * 2); a = take(s.T * s.qd * 2); lse = take(s.seq_rows * 4);
    x_mid = take(s.T * s.d * 2); rstd2 = take(s.T * 4); mn = take(s.T * s.d * 2);
    gu = take(keep ? s.T * 2 * s.f * 2 : 0); act = take(s.T * s.f * 2);      // gate and up: for a backward pass alone
    bytes = o;
  }
};
// keep: one part per block, then the final norm's input and rstd, the temporary and the rotary angles; otherwise two parts used in turn.
struct Arena {
  BlockLayout b;
  size_t parts, x_last, rstd_f, tmp, rope, total;
  Arena(const Sizes& s, int n_layers, bool keep) : b(s, keep) {
    parts = keep ? n_layers : (n_layers < 2 ? n_layers : 2);
    x_last = parts * b.bytes;
    rstd_f = x_last + align256(s.T * s.d * 2);
    tmp = rstd_f + align256(s.T * 4);
    rope = tmp + align256(s.T * s.d * 2);
    total = rope + align256(s.T * s.hd / 2 * sizeof(float2));
  }
};
struct Scratch {
  size_t dhz, dx, dgu, dn, da, dqkv, dsum, total;
  explicit Scratch(const Sizes& s) {
    size_t o = 0;
    auto take = [&](size_t n) { const size_t at = o; o += align256(n); return at; };
    dhz = take(s.T * s.d * 2); dx = take(s.T * s.d * 2); dgu = take(s.T * 2 * s.f * 2);
    dn = take(s.T * s.d * 2); da = take(s.T * s.qd * 2); dqkv = take(s.T * s.qkv * 2); dsum = take(s.seq_rows * 4 * (s.hd / 16));
    total = o;
  }
};

// Y[T, O] = X[T, K] W[O, K]^T, or with w_rows_contract: Y[T, O] = X[T, K] W[K, O]
int product(faar_ctx* ctx, size_t T, int O, int K, const void* X, int64_t ldx, const void* W, int64_t ldw, bool w_rows_contract,
            void* Y, int64_t ldy, void* ws) {
  faar_gemm_args a = {};
  a.mode = FAAR_GEMM_REF;
  a.M = (int)T; a.N = O; a.Kc = K;
  a.A = X; a.lda = ldx;
  a.B = W; a.ldb = ldw; a.b_mn = w_rows_contract;
  a.status = reinterpret_cast<uint32_t*>(ws);
  a.Yout = Y; a.yout_dtype = FAAR_BF16; a.ldy = ldy;
  return faar_launch_gemm(ctx, &a, nullptr);
}

// [gate | up] = X W^T over the stacked weights and act = silu(gate) up; gu null: act alone
int product_gated(faar_ctx* ctx, size_t T, int f, int K, const void* X, const void* W, void* gu, void* act, void* ws) {
  faar_gemm_args a = {};
  a.mode = FAAR_GEMM_REF;
  a.M = (int)T; a.N = 2 * f; a.Kc = K;
  a.A = X; a.lda = K;
  a.B = W; a.ldb = K;
  a.whole = 1;
  a.status = reinterpret_cast<uint32_t*>(ws);
  a.Yout = gu; a.yout_dtype = FAAR_BF16; a.ldy = 2 * f;
  a.gated = FAAR_GATED_FWD; a.act = act;
  return faar_launch_gemm(ctx, &a, nullptr);
}
// [q | k | v] = X W^T over the stacked weights, the heads of q and k turned by their row's angles
int product_rope(faar_ctx* ctx, const faar_model* m, const Sizes& s, const void* X, const void* W, const float2* rope, void* qkv, void* ws) {
  faar_gemm_args a = {};
  a.mode = FAAR_GEMM_REF;
  a.M = (int)s.T; a.N = s.qkv; a.Kc = s.d;
  a.A = X; a.lda = s.d;
  a.B = W; a.ldb = s.d;
  a.whole = 1;
  a.status = reinterpret_cast<uint32_t*>(ws);
  a.Yout = qkv; a.yout_dtype = FAAR_BF16; a.ldy = s.qkv;
  a.rope = rope; a.rope_cols = s.qd + s.kvd; a.head_dim = m->head_dim;
  return faar_launch_gemm(ctx, &a, nullptr);
}
// [d gate | d up] of act = silu(gate) up from d act = dY[T, K] W[K, f] (which is not kept) and the forward pass's [gate | up]
int product_gated_bwd(faar_ctx* ctx, size_t T, int f, int K, const void* dY, const void* W, const void* gu, void* dgu, void* ws) {
  faar_gemm_args a = {};
  a.mode = FAAR_GEMM_REF;
  a.M = (int)T; a.N = f; a.Kc = K;
  a.A = dY; a.lda = K;
  a.B = W; a.ldb = f; a.b_mn = 1;
  a.whole = 1;
  a.status = reinterpret_cast<uint32_t*>(ws);
  a.Yout = dgu; a.yout_dtype = FAAR_BF16; a.ldy = 2 * f;
  a.gated = FAAR_GATED_BWD; a.gate_up = gu;
  return faar_launch_gemm(ctx, &a, nullptr);
}

// dA = dY W_o, the gradient of the attention output a, and the row sums of dA * a by head (*parts of them).  Up to 128 rows such a
// product is better the other way round (see faar_launch_gemm), without them: *parts = 0.
int product_sums(faar_ctx* ctx, const Sizes& s, const void* dY, const void* W, const void* a_out, void* dA, float* sums, int* parts, void* ws) {
  *parts = 0;
  if (s.T <= 128) return product(ctx, s.T, s.qd, s.d, dY, s.d, W, s.qd, true, dA, s.qd, ws);
  faar_gemm_args a = {};
  a.mode = FAAR_GEMM_REF;
  a.M = (int)s.T; a.N = s.qd; a.Kc = s.d;
  a.A = dY; a.lda = s.d;
  a.B = W; a.ldb = s.qd; a.b_mn = 1;
  a.status = reinterpret_cast<uint32_t*>(ws);
  a.Yout = dA; a.yout_dtype = FAAR_BF16; a.ldy = s.qd;
  a.sum_with = a_out; a.sums = sums; a.sum_dim = s.hd; a.sum_parts = parts;
  return faar_launch_gemm(ctx, &a, nullptr);
}

// Logits and, if wanted, their rows' softmax statistics at temperature tau
struct Stats { float tau; void* out; size_t bytes; };
int product_logits(faar_ctx* ctx, const faar_model* m, size_t T, const void* H, void* Z, const Stats& st, void* ws) {
  if (!st.out) return product(ctx, T, m->vocab, m->hidden, H, m->hidden, m->lm_head, m->hidden, false, Z, m->vocab, ws);
  faar_gemm_args a = {};
  a.mode = FAAR_GEMM_REF;
  a.M = (int)T; a.N = m->vocab; a.Kc = m->hidden;
  a.A = H; a.lda = m->hidden;
  a.B = m->lm_head; a.ldb = m->hidden;
  a.whole = 1;
  a.status = reinterpret_cast<uint32_t*>(ws);
  a.Yout = Z; a.yout_dtype = FAAR_BF16; a.ldy = m->vocab;
  a.stats = reinterpret_cast<float2*>(st.out);
  a.stats_c = (float)(1.4426950408889634 / (double)st.tau);
  return faar_launch_gemm(ctx, &a, nullptr);
}

int group_rows(const faar_linear_group& g) {
  int r = 0;
  for (int i = 0; i < g.n; ++i) r += g.lin[i].rows;
  return r;
}
int segments(const faar_linear_group& g, faar_bwd_state (&seg)[FAAR_MAX_SEGMENTS]) {
  for (int i = 0; i < g.n; ++i) {
    const faar_linear& l = g.lin[i];
    seg[i] = {l.V, l.code, l.scales, l.s_global, l.adam_m, l.adam_u, l.dV, 0.f, l.rows};
  }
  return g.n;
}
// A group's soft weights as items of a launch; returns how many.
int soft_items(const faar_linear_group& g, int K, faar_soft_item* item) {
  __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(g.Wsoft);
  for (int i = 0; i < g.n; ++i) {
    const faar_linear& l = g.lin[i];
    item[i] = {l.V, l.code, l.scales, l.s_global, out, (int64_t)l.rows * K};
    out += (int64_t)l.rows * K;
  }
  return g.n;
}
// Soft weights of the blocks from l on in one launch, as many whole blocks as SOFT_AHEAD weights allow; returns their
// number in *n.  0: the next block is larger than that, and its groups' soft weights are formed just before their products,
// which then find them in L2.  A small model is a chain of launches of a few microseconds: an alignment step of two 128-wide
// blocks 321 -> 310 us.
constexpr int64_t SOFT_AHEAD = 16 << 20;        // 32 MB of BF16, which stays in L2 until used
int soft_blocks(faar_ctx* ctx, const faar_model* m, const Sizes& s, int l, float beta, int* n) {
  const int64_t per_block = (int64_t)s.d * (s.qkv + s.qd + 3 * (int64_t)s.f);
  constexpr int PER_BLOCK = 7;
  faar_soft_item item[FAAR_MAX_SOFT_ITEMS];
  int items = 0;
  for (*n = 0; l + *n < m->n_layers && items + PER_BLOCK <= FAAR_MAX_SOFT_ITEMS && (*n + 1) * per_block <= SOFT_AHEAD; ++*n) {
    const faar_block& b = m->blocks[l + *n];
    items += soft_items(b.qkv, s.d, item + items);
    items += soft_items(b.o, s.qd, item + items);
    items += soft_items(b.gate_up, s.d, item + items);
    items += soft_items(b.down, s.f, item + items);
  }
  return items ? faar_launch_soft_weights(ctx, items, item, beta) : 0;
}
// A group's operand: frozen weights, soft weights (formed already), or soft weights formed first.
enum Weights { FROZEN, SOFT, FORM_SOFT };
int group_operand(faar_ctx* ctx, const faar_linear_group& g, int K, Weights weights, float beta, const void** W) {
  *W = weights == FROZEN ? g.W : g.Wsoft;
  if (weights != FORM_SOFT) return 0;
  faar_soft_item item[FAAR_MAX_SEGMENTS];
  const int n = soft_items(g, K, item);
  return faar_launch_soft_weights(ctx, n, item, beta);
}
int group_forward(faar_ctx* ctx, const faar_linear_group& g, size_t T, int K, const void* X, Weights weights, float beta, void* Y, void* ws) {
  const int rows = group_rows(g);
  const void* W;
  const int e = group_operand(ctx, g, K, weights, beta, &W);
  return e ? e : product(ctx, T, rows, K, X, K, W, K, false, Y, rows, ws);
}
// A group's backward: the gradient towards the common input, then the update of every V (at the pre-update soft weights).
int group_update(faar_ctx* ctx, const faar_linear_group& g, size_t T, int K, const void* dY, const void* X, const faar_hparams* hp, void* ws,
                 bool beside = true);
int group_backward(faar_ctx* ctx, const faar_linear_group& g, size_t T, int K, const void* dY, const void* X, const faar_hparams* hp,
                   void* dX, void* ws) {
  const int rows = group_rows(g);
  const int e = product(ctx, T, K, rows, dY, rows, g.Wsoft, K, true, dX, K, ws);
  return e ? e : group_update(ctx, g, T, K, dY, X, hp, ws);
}
int group_update(faar_ctx* ctx, const faar_linear_group& g, size_t T, int K, const void* dY, const void* X, const faar_hparams* hp, void* ws,
                 bool beside) {
  const int rows = group_rows(g);
  faar_bwd_state seg[FAAR_MAX_SEGMENTS];
  const int n = segments(g, seg);
  return faar_bwd_group(ctx, n, seg, (int)T, K, hp, dY, rows, X, K, ws, beside);
}

constexpr size_t OVERLAP_LIMIT = 28 << 20;     // see faar_model_overlap

bool aligned(const void* p) { return p && (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// The checks of the single entry points (faar_embedding, faar_rmsnorm, faar_rope, faar_layer_ref, faar_layer_bwd_rowmajor
// and so on) for everything that a pass hands to their kernels.
bool sizes_ok(const faar_model* m) {
  if (m->n_layers <= 0 || m->hidden <= 0 || m->ffn <= 0 || m->n_heads <= 0 || m->n_kv_heads <= 0 || m->head_dim <= 0) return false;
  // widths are held as int, and the dW epilogue counts up to 7 rows of V in 32 bits
  const long long q = (long long)m->n_heads * m->head_dim, kv = (long long)m->n_kv_heads * m->head_dim;
  return q + 2 * kv <= 0x7FFFFFFFll && 8 * q <= 0x7FFFFFFFll && 8ll * m->ffn <= 0x7FFFFFFFll && 8ll * m->hidden <= 0x7FFFFFFFll;
}
int check_group(const faar_linear_group& g, int n, const int* rows, bool quantised, const faar_hparams* hp) {
  if (g.n != n) return FAAR_ERR_INVALID_ARG;
  if (quantised ? !aligned(g.Wsoft) : !aligned(g.W)) return g.W || g.Wsoft ? FAAR_ERR_ALIGN : FAAR_ERR_INVALID_ARG;
  for (int i = 0; i < n; ++i) {
    const faar_linear& l = g.lin[i];
    if (l.rows != rows[i]) return FAAR_ERR_SHAPE;
    if (!quantised) continue;
    if (!l.V || !l.code || !l.scales || !l.s_global) return FAAR_ERR_INVALID_ARG;
    if (hp && hp->opt == 1 && (!l.adam_m || !l.adam_u)) return FAAR_ERR_INVALID_ARG;
    if (!aligned(l.V) || !aligned(l.code) || (l.adam_m && !aligned(l.adam_m)) || (l.adam_u && !aligned(l.adam_u)) ||
        (l.dV && !aligned(l.dV)))
      return FAAR_ERR_ALIGN;
  }
  return FAAR_OK;
}
int check_model(const faar_ctx* ctx, const faar_model* m, int batch, int seq, bool quantised, const faar_hparams* hp, const void* ws,
                size_t ws_bytes) {
  if (!ctx || !m || !m->blocks || !m->embed || !m->lm_head || !m->final_norm) return FAAR_ERR_INVALID_ARG;
  if (!(m->eps >= 0.f) || !isfinite(m->eps) || !(m->theta > 1.f) || !isfinite(m->theta)) return FAAR_ERR_INVALID_ARG;
  if (batch <= 0 || seq <= 0 || (long long)batch * seq > 0x7FFFFFFFll || !sizes_ok(m) || m->n_heads % m->n_kv_heads ||
      (m->head_dim != 64 && m->head_dim != 128))
    return FAAR_ERR_SHAPE;
  if (m->vocab <= 0 || m->vocab % 16 || m->hidden % 16 || m->ffn % 16) return FAAR_ERR_SHAPE;
  if (!aligned(m->embed) || !aligned(m->lm_head) || !aligned(m->final_norm)) return FAAR_ERR_ALIGN;
  if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < FAAR_WS_HEADER + 2 * sizeof(float) * FAAR_MAX_PARTIALS)
    return FAAR_ERR_WORKSPACE;
  const int qd = m->n_heads * m->head_dim, kvd = m->n_kv_heads * m->head_dim;
  const int qkv[3] = {qd, kvd, kvd}, one[1] = {m->hidden}, gu[2] = {m->ffn, m->ffn};
  for (int l = 0; l < m->n_layers; ++l) {
    const faar_block& b = m->blocks[l];
    if (!b.attn_norm || !b.mlp_norm) return FAAR_ERR_INVALID_ARG;
    if (!aligned(b.attn_norm) || !aligned(b.mlp_norm)) return FAAR_ERR_ALIGN;
    int st = check_group(b.qkv, 3, qkv, quantised, hp);
    if (!st) st = check_group(b.o, 1, one, quantised, hp);
    if (!st) st = check_group(b.gate_up, 2, gu, quantised, hp);
    if (!st) st = check_group(b.down, 1, one, quantised, hp);
    if (st) return st;
  }
  return FAAR_OK;
}

// The first block's input and norm and the rotary angles, into the arena of a pass.
int begin(faar_ctx* ctx, const faar_model* m, int batch, int seq, const int* tokens, const int* pos, bool keep, uint8_t* arena) {
  const Sizes s = sizes(m, batch, seq);
  const Arena A(s, m->n_layers, keep);
  return faar_launch_embed_rmsnorm(ctx, (int)s.T, s.d, m->vocab, m->embed, tokens, arena + A.b.x_in, m->blocks[0].attn_norm, m->eps,
                                   arena + A.b.hn, reinterpret_cast<float*>(arena + A.b.rstd1), pos, s.hd, m->theta,
                                   reinterpret_cast<float2*>(arena + A.rope));
}
// The blocks, the final norm and the LM head.  begun: the arena that begin() has filled, this pass's or that of another pass
// (which keeps its activations) on the same tokens.
int forward(faar_ctx* ctx, const faar_model* m, int batch, int seq, bool quantised, float beta, bool keep, uint8_t* arena,
            const uint8_t* begun, void* Z, void* Hout, const Stats& stats, void* ws) {
  const Sizes s = sizes(m, batch, seq);
  const Arena A(s, m->n_layers, keep);
  const int T = (int)s.T;
  auto part = [&](int l) { return arena + (keep ? l : l % (int)A.parts) * A.b.bytes; };
  uint8_t* const tmp = arena + A.tmp;
  uint8_t* p = nullptr;
  const float2* const rope = reinterpret_cast<const float2*>(begun + Arena(s, m->n_layers, keep || begun != arena).rope);
  int e = 0;
  int soft_end = 0;                              // blocks below this have their soft weights
  for (int l = 0; l < m->n_layers && !e; ++l) {
    const faar_block& b = m->blocks[l];
    p = part(l);
    if (quantised && l >= soft_end) {
      int n = 0;
      e = soft_blocks(ctx, m, s, l, beta, &n);
      if (e) break;
      soft_end = l + n;
    }
    const Weights w = !quantised ? FROZEN : (l < soft_end ? SOFT : FORM_SOFT);
    __nv_bfloat16* const qkv = reinterpret_cast<__nv_bfloat16*>(p + A.b.qkv);
    const void *Wqkv = nullptr, *Wgu = nullptr;
    e = group_operand(ctx, b.qkv, s.d, w, beta, &Wqkv);
    const uint8_t* const in = l == 0 ? begun : p;          // x_in and hn lie first in either form of the arena
    if (!e) e = product_rope(ctx, m, s, in + A.b.hn, Wqkv, rope, qkv, ws);
    if (!e)
      e = faar_launch_attention_fwd(ctx, batch, seq, m->n_heads, m->n_kv_heads, m->head_dim, qkv, s.qkv, qkv + s.qd, qkv + s.qd + s.kvd,
                                    s.qkv, p + A.b.a, s.qd, reinterpret_cast<float*>(p + A.b.lse));
    if (!e) e = group_forward(ctx, b.o, s.T, s.qd, p + A.b.a, w, beta, tmp, ws);
    // residual connection and the MLP's norm in one pass
    if (!e)
      e = faar_launch_rmsnorm(ctx, T, s.d, in + A.b.x_in, s.d, tmp, s.d, p + A.b.x_mid, s.d, b.mlp_norm, m->eps, p + A.b.mn, s.d,
                              reinterpret_cast<float*>(p + A.b.rstd2));
    __nv_bfloat16* const gu = reinterpret_cast<__nv_bfloat16*>(p + A.b.gu);
    // act = silu(gate) up leaves with the product; gate and up themselves only where a backward pass will read them
    if (!e) e = group_operand(ctx, b.gate_up, s.d, w, beta, &Wgu);
    if (!e) e = product_gated(ctx, s.T, s.f, s.d, p + A.b.mn, Wgu, keep ? gu : nullptr, p + A.b.act, ws);
    if (!e) e = group_forward(ctx, b.down, s.T, s.f, p + A.b.act, w, beta, tmp, ws);
    if (e) break;
    // residual connection and the next block's attention norm (after the last block: the final norm)
    const bool last = l + 1 == m->n_layers;
    uint8_t* const n = last ? nullptr : part(l + 1);
    e = faar_launch_rmsnorm(ctx, T, s.d, p + A.b.x_mid, s.d, tmp, s.d, last ? arena + A.x_last : n + A.b.x_in, s.d,
                            last ? m->final_norm : m->blocks[l + 1].attn_norm, m->eps, last ? Hout : n + A.b.hn, s.d,
                            reinterpret_cast<float*>(last ? arena + A.rstd_f : n + A.b.rstd1));
  }
  return e ? e : product_logits(ctx, m, s.T, Hout, Z, stats, ws);
}

int backward(faar_ctx* ctx, const faar_model* m, int batch, int seq, const int* pos, const faar_hparams* hp, uint8_t* arena,
             const void* dZ, int64_t ldz, const void* dH, uint8_t* scratch, void* ws) {
  const Sizes s = sizes(m, batch, seq);
  const Arena A(s, m->n_layers, true);
  const Scratch S(s);
  const int T = (int)s.T;
  uint8_t* const dx = scratch + S.dx;
  // LM head (frozen): dH += dZ W_lm, then the final norm
  int e = product(ctx, s.T, s.d, m->vocab, dZ, ldz, m->lm_head_t, m->ld_lm_head_t, false, scratch + S.dhz, s.d, ws);
  if (!e)
    e = faar_launch_rmsnorm_bwd(ctx, T, s.d, scratch + S.dhz, dH, nullptr, s.d, arena + A.x_last, s.d, m->final_norm,
                                reinterpret_cast<const float*>(arena + A.rstd_f), nullptr, 0, dx, s.d);
  for (int l = m->n_layers - 1; l >= 0 && !e; --l) {
    const faar_block& b = m->blocks[l];
    uint8_t* const p = arena + (size_t)l * A.b.bytes;
    const __nv_bfloat16* const gu = reinterpret_cast<const __nv_bfloat16*>(p + A.b.gu);
    __nv_bfloat16* const dgu = reinterpret_cast<__nv_bfloat16*>(scratch + S.dgu);
    // MLP branch: x = x_mid + act W_down^T
    e = product_gated_bwd(ctx, s.T, s.f, s.d, dx, b.down.Wsoft, gu, dgu, ws);
    if (!e) e = group_backward(ctx, b.gate_up, s.T, s.d, dgu, p + A.b.mn, hp, scratch + S.dn, ws);
    if (!e) e = group_update(ctx, b.down, s.T, s.f, dx, p + A.b.act, hp, ws);       // next to the two before it
    if (!e)
      e = faar_launch_rmsnorm_bwd(ctx, T, s.d, scratch + S.dn, nullptr, nullptr, s.d, p + A.b.x_mid, s.d, b.mlp_norm,
                                  reinterpret_cast<const float*>(p + A.b.rstd2), dx, s.d, dx, s.d);
    // attention branch: x_mid = x_in + a W_o^T
    const __nv_bfloat16* const qkv = reinterpret_cast<const __nv_bfloat16*>(p + A.b.qkv);
    __nv_bfloat16* const dqkv = reinterpret_cast<__nv_bfloat16*>(scratch + S.dqkv);
    // the tcgen05 kernels turn dq and dk back on the way out; the others leave that to a pass over both, which lie side by side
    // and take the row sums of dO * O from the product that forms dO
    const bool turned = ctx->tune_attention_fragments == 0;
    float* const dsum = reinterpret_cast<float*>(scratch + S.dsum);
    int parts = 0;
    if (!e && turned) e = product_sums(ctx, s, dx, b.o.Wsoft, p + A.b.a, scratch + S.da, dsum, &parts, ws);
    if (!e && !turned) e = product(ctx, s.T, s.qd, s.d, dx, s.d, b.o.Wsoft, s.qd, true, scratch + S.da, s.qd, ws);
    if (!e)
      e = faar_launch_attention_bwd(ctx, batch, seq, m->n_heads, m->n_kv_heads, m->head_dim, qkv, s.qkv, qkv + s.qd, qkv + s.qd + s.kvd,
                                    s.qkv, p + A.b.a, scratch + S.da, s.qd, reinterpret_cast<const float*>(p + A.b.lse),
                                    dsum, dqkv, dqkv + s.qd, dqkv + s.qd + s.kvd, turned ? reinterpret_cast<const float2*>(arena + A.rope) : nullptr,
                                    parts);
    if (!e && turned) e = group_update(ctx, b.o, s.T, s.qd, dx, p + A.b.a, hp, ws);          // next to dQ (and so to dK / dV)
    if (!e && !turned) e = group_update(ctx, b.o, s.T, s.qd, dx, p + A.b.a, hp, ws, false);
    if (!e && !turned) e = faar_launch_rope(ctx, T, m->n_heads + m->n_kv_heads, m->head_dim, dqkv, s.qkv, pos, m->theta, 1, dqkv, s.qkv);
    if (!e) e = group_backward(ctx, b.qkv, s.T, s.d, dqkv, p + A.b.hn, hp, scratch + S.dn, ws);
    if (!e)
      e = faar_launch_rmsnorm_bwd(ctx, T, s.d, scratch + S.dn, nullptr, nullptr, s.d, p + A.b.x_in, s.d, b.attn_norm,
                                  reinterpret_cast<const float*>(p + A.b.rstd1), dx, s.d, dx, s.d);
  }
  return e;
}

// Both forward passes at once: the frozen one on the context's side stream, between two events, behind the first block's
// input and norm, which they share.  The products of either use nothing of the workspace but its status word.
int forward_both(faar_ctx* ctx, const faar_model* m, int batch, int seq, const int* tokens, const int* pos, float beta, uint8_t* arena_fp,
                 void* Z_fp, void* H_fp, uint8_t* arena, void* Z, void* H, const Stats& stats_fp, const Stats& stats, void* ws) {
  cudaError_t ce = cudaSuccess;
  if (!ctx->side_stream) ce = cudaStreamCreateWithFlags(&ctx->side_stream, cudaStreamNonBlocking);
  if (ce == cudaSuccess && !ctx->ev_fork) ce = cudaEventCreateWithFlags(&ctx->ev_fork, cudaEventDisableTiming);
  if (ce == cudaSuccess && !ctx->ev_join) ce = cudaEventCreateWithFlags(&ctx->ev_join, cudaEventDisableTiming);
  if (ce != cudaSuccess) return (int)ce;
  int e = begin(ctx, m, batch, seq, tokens, pos, true, arena);
  if (e) return e;
  const cudaStream_t main = ctx->stream;
  ce = cudaEventRecord(ctx->ev_fork, main);
  if (ce == cudaSuccess) ce = cudaStreamWaitEvent(ctx->side_stream, ctx->ev_fork, 0);
  if (ce != cudaSuccess) return (int)ce;
  ctx->stream = ctx->side_stream;
  e = forward(ctx, m, batch, seq, false, beta, false, arena_fp, arena, Z_fp, H_fp, stats_fp, ws);
  ctx->stream = main;
  // joined whatever happened, so that the caller's stream orders everything that was enqueued
  ce = cudaEventRecord(ctx->ev_join, ctx->side_stream);
  if (!e) e = forward(ctx, m, batch, seq, true, beta, true, arena, arena, Z, H, stats, ws);
  if (ce == cudaSuccess) ce = cudaStreamWaitEvent(main, ctx->ev_join, 0);
  return e ? e : (int)ce;
}

// The context's device is current for the duration of a call.
struct Device {
  int prev = -1, err = 0;
  explicit Device(int dev) {
    cudaError_t e = cudaGetDevice(&prev);
    if (e == cudaSuccess && prev != dev) e = cudaSetDevice(dev); else if (e == cudaSuccess) prev = -1;
    if (e != cudaSuccess) { err = (int)e; prev = -1; }
  }
  ~Device() { if (prev >= 0) (void)cudaSetDevice(prev); }
};
int status(faar_ctx* ctx, int e) {
  if (e == 0) return FAAR_OK;
  ctx->last_cuda_error = e;
  return FAAR_ERR_CUDA;
}

}  // namespace

extern "C" {

int faar_model_sizes(const faar_model* m, int batch, int seq, int keep, size_t* arena_bytes, size_t* scratch_bytes) {
  if (!m || !arena_bytes || !scratch_bytes) return FAAR_ERR_INVALID_ARG;
  if (batch <= 0 || seq <= 0 || !sizes_ok(m)) return FAAR_ERR_SHAPE;
  const Sizes s = sizes(m, batch, seq);
  *arena_bytes = Arena(s, m->n_layers, keep != 0).total;
  *scratch_bytes = Scratch(s).total;
  return FAAR_OK;
}

static int check_stats(faar_ctx* ctx, const faar_model* m, int batch, int seq, const Stats& st) {
  if (!st.out) return FAAR_OK;
  if (!(st.tau > 0.f) || !isfinite(st.tau)) return FAAR_ERR_INVALID_ARG;
  return faar_check_logit_stats(ctx, batch * seq, m->vocab, st.out, st.bytes);
}
static int model_forward(faar_ctx* ctx, const faar_model* m, int batch, int seq, const int* tokens, const int* positions, int quantised,
                         float beta, int keep, void* arena, size_t arena_bytes, void* Z, void* H, const Stats& stats, void* workspace,
                         size_t workspace_bytes) {
  int st = check_model(ctx, m, batch, seq, quantised != 0, nullptr, workspace, workspace_bytes);
  if (st) return st;
  if (!tokens || !positions || !arena || !Z || !H) return FAAR_ERR_INVALID_ARG;
  if (quantised && (!(beta > 0.f) || !isfinite(beta))) return FAAR_ERR_INVALID_ARG;
  if (!aligned(Z) || !aligned(H) || (reinterpret_cast<uintptr_t>(arena) & 255u)) return FAAR_ERR_ALIGN;
  size_t need = 0, scratch = 0;
  if ((st = faar_model_sizes(m, batch, seq, keep, &need, &scratch))) return st;
  if (arena_bytes < need) return FAAR_ERR_WORKSPACE;
  if ((st = check_stats(ctx, m, batch, seq, stats))) return st;
  Device dev(ctx->device);
  if (dev.err) return status(ctx, dev.err);
  uint8_t* const at = reinterpret_cast<uint8_t*>(arena);
  const int e = begin(ctx, m, batch, seq, tokens, positions, keep != 0, at);
  return status(ctx, e ? e : forward(ctx, m, batch, seq, quantised != 0, beta, keep != 0, at, at, Z, H, stats, workspace));
}
int faar_model_forward(faar_ctx* ctx, const faar_model* m, int batch, int seq, const int* tokens, const int* positions, int quantised,
                       float beta, int keep, void* arena, size_t arena_bytes, void* Z, void* H, void* workspace,
                       size_t workspace_bytes) {
  return model_forward(ctx, m, batch, seq, tokens, positions, quantised, beta, keep, arena, arena_bytes, Z, H, {1.f, nullptr, 0}, workspace,
                       workspace_bytes);
}
int faar_model_forward_stats(faar_ctx* ctx, const faar_model* m, int batch, int seq, const int* tokens, const int* positions, int quantised,
                             float beta, int keep, void* arena, size_t arena_bytes, void* Z, void* H, float tau, void* stats, size_t stats_bytes, void* workspace,
                             size_t workspace_bytes) {
  if (!stats) return FAAR_ERR_INVALID_ARG;
  return model_forward(ctx, m, batch, seq, tokens, positions, quantised, beta, keep, arena, arena_bytes, Z, H, {tau, stats, stats_bytes}, workspace,
                       workspace_bytes);
}

// Overlap pays while the passes are chains of launches that leave much of the GPU idle.  Whole alignment step, one pass after
// the other -> both at once, by tokens x widest product: 0.1 M 312 -> 248 us, 0.5 M 428 -> 356, 2.1 M 607 -> 525, 8.4 M
// 1060 -> 998, 16.8 M 1491 -> 1457, 24.6 M 3206 -> 3146, 33.6 M 3000 -> 3010 and 67 M 5305 -> 5330, where every product
// fills the GPU (and both arenas at once are gigabytes).
int faar_model_overlap(const faar_model* m, int batch, int seq, int* overlap) {
  if (!m || !overlap) return FAAR_ERR_INVALID_ARG;
  if (batch <= 0 || seq <= 0 || !sizes_ok(m)) return FAAR_ERR_SHAPE;
  const Sizes s = sizes(m, batch, seq);
  const size_t widest = s.qkv > 2 * s.f ? s.qkv : 2 * s.f;
  *overlap = s.T * widest <= OVERLAP_LIMIT;
  return FAAR_OK;
}

static int model_forward_both(faar_ctx* ctx, const faar_model* m, int batch, int seq, const int* tokens, const int* positions, float beta,
                              void* arena_fp, size_t arena_fp_bytes, void* Z_fp, void* H_fp, void* arena, size_t arena_bytes, void* Z, void* H,
                              const Stats& stats_fp, const Stats& stats, void* workspace, size_t workspace_bytes) {
  int st = check_model(ctx, m, batch, seq, false, nullptr, workspace, workspace_bytes);
  if (!st) st = check_model(ctx, m, batch, seq, true, nullptr, workspace, workspace_bytes);
  if (st) return st;
  if (!tokens || !positions || !arena_fp || !Z_fp || !H_fp || !arena || !Z || !H || !(beta > 0.f) || !isfinite(beta)) return FAAR_ERR_INVALID_ARG;
  if (!aligned(Z_fp) || !aligned(H_fp) || !aligned(Z) || !aligned(H) || (reinterpret_cast<uintptr_t>(arena) & 255u) ||
      (reinterpret_cast<uintptr_t>(arena_fp) & 255u))
    return FAAR_ERR_ALIGN;
  size_t need_fp = 0, need = 0, scratch = 0;
  if ((st = faar_model_sizes(m, batch, seq, 0, &need_fp, &scratch))) return st;
  if ((st = faar_model_sizes(m, batch, seq, 1, &need, &scratch))) return st;
  if (arena_fp_bytes < need_fp || arena_bytes < need) return FAAR_ERR_WORKSPACE;
  if ((st = check_stats(ctx, m, batch, seq, stats_fp)) || (st = check_stats(ctx, m, batch, seq, stats))) return st;
  Device dev(ctx->device);
  if (dev.err) return status(ctx, dev.err);
  return status(ctx, forward_both(ctx, m, batch, seq, tokens, positions, beta, reinterpret_cast<uint8_t*>(arena_fp), Z_fp, H_fp,
                                  reinterpret_cast<uint8_t*>(arena), Z, H, stats_fp, stats, workspace));
}

int faar_model_forward_both(faar_ctx* ctx, const faar_model* m, int batch, int seq, const int* tokens, const int* positions, float beta,
                            void* arena_fp, size_t arena_fp_bytes, void* Z_fp, void* H_fp, void* arena, size_t arena_bytes, void* Z,
                            void* H, void* workspace, size_t workspace_bytes) {
  return model_forward_both(ctx, m, batch, seq, tokens, positions, beta, arena_fp, arena_fp_bytes, Z_fp, H_fp, arena, arena_bytes, Z, H,
                            {1.f, nullptr, 0}, {1.f, nullptr, 0}, workspace, workspace_bytes);
}
int faar_model_forward_both_stats(faar_ctx* ctx, const faar_model* m, int batch, int seq, const int* tokens, const int* positions, float beta,
                                  void* arena_fp, size_t arena_fp_bytes, void* Z_fp, void* H_fp, void* arena, size_t arena_bytes, void* Z,
                                  void* H, float tau, void* stats_fp, void* stats, size_t stats_bytes, void* workspace, size_t workspace_bytes) {
  if (!stats_fp || !stats) return FAAR_ERR_INVALID_ARG;
  return model_forward_both(ctx, m, batch, seq, tokens, positions, beta, arena_fp, arena_fp_bytes, Z_fp, H_fp, arena, arena_bytes, Z, H,
                            {tau, stats_fp, stats_bytes}, {tau, stats, stats_bytes}, workspace, workspace_bytes);
}

int faar_model_backward(faar_ctx* ctx, const faar_model* m, int batch, int seq, const int* positions, const faar_hparams* hp,
                        void* arena, size_t arena_bytes, const void* dZ, int64_t ldz, const void* dH, void* scratch,
                        size_t scratch_bytes, void* workspace, size_t workspace_bytes) {
  int st = faar_check_hparams(hp, true);
  if (st) return st;
  st = check_model(ctx, m, batch, seq, true, hp, workspace, workspace_bytes);
  if (st) return st;
  if (!positions || !arena || !dZ || !dH || !scratch || !m->lm_head_t) return FAAR_ERR_INVALID_ARG;
  if (ldz < m->vocab || m->ld_lm_head_t < m->vocab) return FAAR_ERR_SHAPE;
  if (!aligned(dZ) || !aligned(dH) || !aligned(m->lm_head_t) || ldz % 8 || m->ld_lm_head_t % 8 || (reinterpret_cast<uintptr_t>(arena) & 255u) ||
      (reinterpret_cast<uintptr_t>(scratch) & 255u))
    return FAAR_ERR_ALIGN;
  size_t need = 0, need_s = 0;
  if ((st = faar_model_sizes(m, batch, seq, 1, &need, &need_s))) return st;
  if (arena_bytes < need || scratch_bytes < need_s) return FAAR_ERR_WORKSPACE;
  Device dev(ctx->device);
  if (dev.err) return status(ctx, dev.err);
  if (ctx->wsoft_ws == workspace) ctx->wsoft_ws = nullptr;
  return status(ctx, backward(ctx, m, batch, seq, positions, hp, reinterpret_cast<uint8_t*>(arena), dZ, ldz, dH,
                              reinterpret_cast<uint8_t*>(scratch), workspace));
}

}  // extern "C"
