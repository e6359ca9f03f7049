"""The passes of a model against the same passes strung together from the library's single calls: what a pass's products do
in their epilogues (the gated product and its backward, rotary embedding) has to give the values of the element-wise calls, over token counts and
widths that fill no tile, one tile, several, and over the width choices of the launches."""
import pytest
import torch

from paper_2603_22370_b200 import faar, stage2

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    from paper_2603_22370_b200 import build
    build.build()
    c = faar.Context(0)
    yield c
    torch.cuda.synchronize()
    c.close()


def make_model(ctx, batch, seq, **cfg):
    cfg = stage2.ModelConfig(**cfg)
    gen = torch.Generator(device=DEV).manual_seed(5)

    def bf(*shape, sigma):
        return (torch.randn(shape, device=DEV, generator=gen) * sigma).to(torch.bfloat16)

    def ones(n):
        return 0.8 + 0.4 * torch.rand(n, device=DEV, generator=gen)

    params = {"embed": bf(cfg.vocab, cfg.hidden, sigma=1.0), "lm_head": bf(cfg.vocab, cfg.hidden, sigma=cfg.hidden**-0.5),
              "final_norm": ones(cfg.hidden)}
    for l in range(cfg.n_layers):
        params[f"attn_norm.{l}"], params[f"mlp_norm.{l}"] = ones(cfg.hidden), ones(cfg.hidden)
    weights = [{n: bf(o, k, sigma=k**-0.5) for n, (o, k) in cfg.linear_shapes().items()} for _ in range(cfg.n_layers)]
    model = stage2.Stage2Model(ctx, cfg, params, weights, batch, seq)
    for layer in model.lin:
        for lin in layer.values():
            lin.V.add_(torch.randn(lin.V.shape, device=DEV, generator=gen) * 0.2).clamp_(0.0, 1.0)
    model.ws = torch.empty(faar.workspace_size(faar.make_shape(max(2 * cfg.ffn, cfg.vocab, 4 * cfg.hidden), max(cfg.ffn, 4 * cfg.hidden), batch * seq)),
                           dtype=torch.uint8, device=DEV)              # room for every single call
    faar.workspace_init(ctx, model.ws)
    tokens = torch.randint(0, cfg.vocab, (batch * seq,), dtype=torch.int32, device=DEV, generator=gen)
    return model, tokens, gen


def empty(*shape, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device=DEV)


def linear(m, X, W):
    Y = empty(X.shape[0], W.shape[0])
    faar.layer_ref(m.ctx, faar.make_shape(W.shape[0], W.shape[1], X.shape[0]), X, W, Y, m.ws)
    return Y


def forward(m, tokens, soft):
    """The calls of one forward pass; returns Z, H and what a backward pass needs."""
    c, ctx, T, d, f = m.cfg, m.ctx, m.T, m.cfg.hidden, m.cfg.ffn
    qd, kvd = c.n_heads * c.head_dim, c.n_kv_heads * c.head_dim
    x, saved = empty(T, d), []
    faar.embedding(ctx, T, d, c.vocab, m.params["embed"], d, tokens, x, d)
    for l in range(c.n_layers):
        g = m.wsoft_group[l] if soft else m.w_group[l]
        W = {n: (m.lin[l][n].Wsoft if soft else m.lin[l][n].W) for n in ("o_proj", "down_proj")}
        s = {"x_in": x, "rstd1": empty(T, dtype=torch.float32), "rstd2": empty(T, dtype=torch.float32),
             "lse": empty(T * c.n_heads, dtype=torch.float32)}
        s["hn"], s["mn"], s["x_mid"], s["a"], s["act"], x_next = empty(T, d), empty(T, d), empty(T, d), empty(T, qd), empty(T, f), empty(T, d)
        faar.rmsnorm(ctx, T, d, x, d, m.params[f"attn_norm.{l}"], c.eps, s["hn"], d, s["rstd1"])
        qkv = s["qkv"] = linear(m, s["hn"], g["qkv"])
        ld = qkv.shape[1]
        faar.rope(ctx, T, c.n_heads + c.n_kv_heads, c.head_dim, qkv, ld, m.pos, c.theta, 0, qkv, ld)
        faar.attention_fwd(ctx, m.batch, m.seq, c.n_heads, c.n_kv_heads, c.head_dim, qkv, ld, qkv[:, qd:], qkv[:, qd + kvd:], ld, s["a"], qd,
                           s["lse"])
        faar.add(ctx, T, d, x, d, linear(m, s["a"], W["o_proj"]), d, s["x_mid"], d)
        faar.rmsnorm(ctx, T, d, s["x_mid"], d, m.params[f"mlp_norm.{l}"], c.eps, s["mn"], d, s["rstd2"])
        gu = s["gu"] = linear(m, s["mn"], g["gate_up"])
        faar.silu_mul(ctx, T, f, gu, 2 * f, gu[:, f:], 2 * f, s["act"], f)
        faar.add(ctx, T, d, s["x_mid"], d, linear(m, s["act"], W["down_proj"]), d, x_next, d)
        x = x_next
        saved.append(s)
    H, rstd = empty(T, d), empty(T, dtype=torch.float32)
    faar.rmsnorm(ctx, T, d, x, d, m.params["final_norm"], c.eps, H, d, rstd)
    return linear(m, H, m.params["lm_head"]), H, (saved, x, rstd)


def backward(m, dZ, dH, kept, hp):
    """The calls of one backward pass on the soft weights; returns {(l, name): dV} (V itself stays)."""
    c, ctx, T, d, f = m.cfg, m.ctx, m.T, m.cfg.hidden, m.cfg.ffn
    qd, kvd, grads = c.n_heads * c.head_dim, c.n_kv_heads * c.head_dim, {}
    saved, x_last, rstd_f = kept

    def towards_input(dY, W):
        dX = empty(T, W.shape[1])
        faar.layer_dx_operand(ctx, faar.make_shape(W.shape[0], W.shape[1], T), dY, W, dX, m.ws)
        return dX

    def update(l, name, dY, X):
        lin = m.lin[l][name]
        g = grads[l, name] = empty(lin.O, lin.K, dtype=torch.float32)
        faar.layer_bwd_rowmajor(ctx, faar.make_shape(lin.O, lin.K, T, ldy=dY.stride(0)), hp, dY, X, lin.V.clone(), lin.code, lin.scales,
                                lin.s_global, lin.m.clone(), lin.u.clone(), g, m.ws)

    def norm_bwd(dy, x, g, rstd, add):
        dx = empty(T, d)
        faar.rmsnorm_bwd(ctx, T, d, dy, d, x, d, g, rstd, add, d, dx, d)
        return dx

    dx = empty(T, d)
    faar.rmsnorm_bwd_sum(ctx, T, d, towards_input(dZ, m.params["lm_head"]), dH, None, d, x_last, d, m.params["final_norm"], rstd_f, None, 0, dx, d)
    for l in reversed(range(c.n_layers)):
        s, g = saved[l], m.wsoft_group[l]
        dact, dgu = towards_input(dx, m.lin[l]["down_proj"].Wsoft), empty(T, 2 * f)
        update(l, "down_proj", dx, s["act"])
        faar.silu_mul_bwd(ctx, T, f, dact, f, s["gu"], 2 * f, s["gu"][:, f:], 2 * f, dgu, 2 * f, dgu[:, f:], 2 * f)
        update(l, "gate_proj", dgu, s["mn"])
        update(l, "up_proj", dgu[:, f:], s["mn"])
        dx = norm_bwd(towards_input(dgu, g["gate_up"]), s["x_mid"], m.params[f"mlp_norm.{l}"], s["rstd2"], dx)
        update(l, "o_proj", dx, s["a"])
        da, qkv = towards_input(dx, m.lin[l]["o_proj"].Wsoft), s["qkv"]
        ld = qkv.shape[1]
        dqkv, dsum = empty(T, ld), empty(T * c.n_heads, dtype=torch.float32)
        faar.attention_bwd(ctx, m.batch, m.seq, c.n_heads, c.n_kv_heads, c.head_dim, qkv, ld, qkv[:, qd:], qkv[:, qd + kvd:], ld, s["a"], da, qd,
                           s["lse"], dsum, dqkv, dqkv[:, qd:], dqkv[:, qd + kvd:])
        faar.rope(ctx, T, c.n_heads + c.n_kv_heads, c.head_dim, dqkv, ld, m.pos, c.theta, 1, dqkv, ld)
        for i, n in enumerate(("q_proj", "k_proj", "v_proj")):
            update(l, n, dqkv[:, (0, qd, qd + kvd)[i]:], s["hn"])
        dx = norm_bwd(towards_input(dqkv, g["qkv"]), s["x_in"], m.params[f"attn_norm.{l}"], s["rstd1"], dx)
    return grads


def rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


@pytest.mark.parametrize("width", [0, 144, 256])
@pytest.mark.parametrize("batch,seq,hidden,heads,kv_heads,head_dim,ffn", [
    (1, 7, 64, 1, 1, 64, 16),             # everything inside one tile; 16 features of the gated product
    (2, 96, 128, 2, 1, 64, 256),
    (3, 100, 128, 2, 1, 64, 80),          # 160 stacked columns
    (1, 129, 128, 3, 1, 64, 336),         # one row more than half a row block
    (2, 500, 512, 4, 2, 128, 1040),       # ragged rows and features, several tiles
    (5, 512, 256, 2, 2, 128, 5008),       # more tiles than CTA pairs: half-width tiles, a narrow last column
])
def test_a_models_passes_are_those_of_its_single_calls(ctx, batch, seq, hidden, heads, kv_heads, head_dim, ffn, width):
    m, tokens, gen = make_model(ctx, batch, seq, vocab=528, hidden=hidden, n_layers=2, n_heads=heads, n_kv_heads=kv_heads, head_dim=head_dim,
                                ffn=ffn)
    tokens[1], tokens[-1] = 528, -1        # outside the table: rows of zeros
    faar.tune_tile_n(ctx, width)
    faar.tune_wide_tiles(ctx, 0)           # every contraction whole, as faar_layer_ref has it: one order of every sum
    try:
        Z_fp, H_fp, _ = m.forward(tokens, quantised=False)
        Z, H, arena = m.forward(tokens, quantised=True, beta=6.0, keep=True)
        dZ, dH = (torch.randn(t.shape, device=DEV, generator=gen).to(torch.bfloat16) for t in (Z, H))
        V0 = {(l, n): m.lin[l][n].V.clone() for l in range(2) for n in stage2.LINEARS}
        hp = faar.make_hparams(beta=6.0, opt=1, lr=5e-4, step=1)
        got = m.backward(dZ, dH, arena, hp, want_dv=True)
        faar.check_status(ctx, m.ws)
        for (l, n), v in V0.items():
            m.lin[l][n].V.copy_(v)
            m.lin[l][n].m.zero_()
            m.lin[l][n].u.zero_()
        Zr_fp, Hr_fp, _ = forward(m, tokens, False)
        Zr, Hr, kept = forward(m, tokens, True)
        want = backward(m, dZ, dH, kept, hp)
    finally:
        faar.tune_tile_n(ctx, 0)
        faar.tune_wide_tiles(ctx, -1)
    assert torch.equal(H_fp, Hr_fp) and torch.equal(Z_fp, Zr_fp) and torch.equal(H, Hr) and torch.equal(Z, Zr)
    worst = max(rel(got[k], want[k]) for k in want)
    # dq and dk turn back before their rounding to BF16, the single calls round before and after: up to 2^-9 of an element, and as
    # much again wherever one of the gradients formed from them (of the norm, gate / up, the attention output) rounds differently
    assert worst <= 4 * 2.0**-9, worst
    assert max(rel(got[1, n], want[1, n]) for n in ("o_proj", "gate_proj", "up_proj", "down_proj")) <= 1e-5      # (before any attention gradient)


@pytest.mark.parametrize("batch,seq,hidden,heads,kv_heads,head_dim,width", [
    (2, 65, 128, 2, 1, 64, 0),            # 16 columns a warp: four parts
    (1, 257, 128, 5, 1, 64, 224),         # tiles that are no whole heads, the last column of half of one
    (1, 128, 192, 3, 1, 64, 0),           # 128 rows: the sums' own launch
    (3, 100, 1024, 3, 3, 128, 0),         # split contraction: eight parts
    (2, 700, 2048, 16, 4, 128, 0),
    (1, 1300, 256, 4, 2, 128, 256),       # whole heads
])
def test_row_sums_of_the_attention_gradient(ctx, batch, seq, hidden, heads, kv_heads, head_dim, width):
    """The sums of dO * O by head leave with the product that forms dO (over 128 rows): in one part a head, in several, of a split contraction."""
    m, tokens, gen = make_model(ctx, batch, seq, vocab=64, hidden=hidden, n_layers=1, n_heads=heads, n_kv_heads=kv_heads, head_dim=head_dim, ffn=64)
    faar.tune_tile_n(ctx, width)
    try:
        Z, H, arena = m.forward(tokens, quantised=True, beta=6.0, keep=True)
        dZ, dH = (torch.randn(t.shape, device=t.device, generator=gen).to(torch.bfloat16) for t in (Z, H))
        V0 = {n: m.lin[0][n].V.clone() for n in stage2.LINEARS}
        hp = faar.make_hparams(beta=6.0, opt=1, lr=5e-4, step=1)
        got = m.backward(dZ, dH, arena, hp, want_dv=True)
        faar.check_status(ctx, m.ws)
        for n, v in V0.items():
            m.lin[0][n].V.copy_(v)
            m.lin[0][n].m.zero_()
            m.lin[0][n].u.zero_()
        _, _, kept = forward(m, tokens, True)
        want = backward(m, dZ, dH, kept, hp)
    finally:
        faar.tune_tile_n(ctx, 0)
    # the bound of the passes' own test, for the gradients that went through the attention's backward pass
    assert max(rel(got[0, n], want[0, n]) for n in ("q_proj", "k_proj", "v_proj")) <= 4 * 2.0**-9
