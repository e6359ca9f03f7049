"""One full-model alignment step (Eq. 6) on the GPU against the Stage-2 oracle, on a small two-block model with
grouped key/value heads: the frozen and the quantised forward passes, the two data terms of the loss, the gradient
towards every one of the 14 rounding tensors, and the state after the update.  Activations are stored in BF16
between the library's calls (the oracle keeps float64), so tensors are compared norm-wise."""
import numpy as np
import pytest
import torch

from oracle import faar_oracle as fo
from oracle import stage2_oracle as so
from paper_2603_22370_b200 import faar, inputs, stage2
from tests.gpu_helpers import DEV, dev_bf16, dev_f32, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2603_22370_b200 import build
    build.build()
    c = faar.Context(0)
    yield c
    torch.cuda.synchronize()
    c.close()


def small_model(seed=0, vocab=512):
    cfg = dict(vocab=vocab, hidden=128, n_layers=2, n_heads=2, n_kv_heads=1, head_dim=64, ffn=256)
    rng = np.random.default_rng(seed)
    bf = inputs.to_bf16_f32
    params = {"embed": bf(rng.standard_normal((cfg["vocab"], cfg["hidden"]))),
              "final_norm": bf(rng.uniform(0.8, 1.2, cfg["hidden"])),
              "lm_head": bf(0.2 * rng.standard_normal((cfg["vocab"], cfg["hidden"])))}
    ocfg = so.ModelCfg(**cfg)
    W_fp, state = [], []
    for l in range(cfg["n_layers"]):
        params[f"attn_norm.{l}"] = bf(rng.uniform(0.8, 1.2, cfg["hidden"]))
        params[f"mlp_norm.{l}"] = bf(rng.uniform(0.8, 1.2, cfg["hidden"]))
        Wl, Sl = {}, {}
        for name, (O, K) in ocfg.linear_shapes().items():
            W = bf(inputs.weights(rng, O, K, sigma=1.0 / np.sqrt(K)))
            scales, sg, code, V0 = fo.softquant_init(W)
            V = np.clip(V0 + 0.1 * rng.standard_normal(V0.shape), 0.02, 0.98).astype(np.float32)
            Wl[name], Sl[name] = W, (V, code, scales, sg)
        W_fp.append(Wl)
        state.append(Sl)
    tokens = rng.integers(0, cfg["vocab"], (2, 96))
    return cfg, ocfg, params, W_fp, state, tokens


def test_stage2_step_matches_the_oracle(ctx):
    cfg, ocfg, params, W_fp, state, tokens = small_model(0)
    B, S = tokens.shape
    dparams = {k: (dev_bf16(v) if k in ("embed", "lm_head") else dev_f32(v)) for k, v in params.items()}
    dweights = [{n: dev_bf16(W_fp[l][n]) for n in so.LINEARS} for l in range(cfg["n_layers"])]
    model = stage2.Stage2Model(ctx, stage2.ModelConfig(**cfg), dparams, dweights, B, S)
    for l in range(cfg["n_layers"]):
        for n in so.LINEARS:
            lin = model.lin[l][n]
            V, code, scales, sg = state[l][n]
            assert np.array_equal(host(lin.code), code) and np.array_equal(host(lin.scales), scales)   # same bracket
            lin.V.copy_(dev_f32(V))
    tok = torch.from_numpy(tokens.reshape(-1).astype(np.int32)).to(DEV)
    beta, tau, lam_kl, lam_r, lr = 6.0, 1.5, 0.7, 0.9, 5e-4
    # ---- forward passes
    Zf, Hf, _ = model.forward(tok, quantised=False)
    Zf_o, Hf_o, _ = so.forward(ocfg, params, W_fp, tokens)
    assert rel_l2(host(Zf), Zf_o) <= 1.5e-2 and rel_l2(host(Hf), Hf_o) <= 1.5e-2
    # ---- the step, with the gradients returned
    res = model.step(tok, beta, tau, lam_kl, lam_r, lr, want_dv=True, fp_outputs=(Zf, Hf))
    Zq, Hq, grads = res["Z_q"], res["H_q"], res["dV"]
    faar.check_status(ctx, model.ws)
    total_o, (l_kl_o, l_mse_o, l_round_o), dV_o = so.stage2_loss_and_grads(ocfg, params, W_fp, state, tokens, beta, tau,
                                                                           lam_kl, lam_r)
    Wq_o = so.quantised_weights(state, beta)
    Zq_o, Hq_o, saved = so.forward(ocfg, params, Wq_o, tokens, keep=True)
    assert rel_l2(host(Zq), Zq_o) <= 1.5e-2 and rel_l2(host(Hq), Hq_o) <= 1.5e-2
    loss = host(model.loss)
    print("L_KL gpu / oracle:", loss[0], l_kl_o, " L_MSE:", loss[1], l_mse_o)
    # The data terms are differences of two nearly equal forward passes: the BF16 storage of Z and H (2^-9 of each
    # pass) is a much larger share of their difference, in the loss values and in the loss gradients alike.
    assert abs(loss[0] - l_kl_o) <= 0.15 * l_kl_o and abs(loss[1] - l_mse_o) <= 0.15 * l_mse_o
    l_round_g = model.round_loss_sum()          # after the update: V has moved by at most lr
    assert abs(l_round_g - l_round_o) <= 4 * lr * 14 + 1e-3 * l_round_o
    # (a) the backward pass on its own: the oracle back-propagates the GPU's own loss gradients
    G = so.backward(ocfg, params, Wq_o, host(res["dZ"]).astype(np.float64), host(res["dH"]).astype(np.float64), saved)
    # (b) the whole step against the oracle's own gradients (looser: the seed noise explained above)
    worst_a, worst_b = 0.0, 0.0
    for l in range(cfg["n_layers"]):
        for n in so.LINEARS:
            V, code, scales, sg = state[l][n]
            Vd = V.astype(np.float64)
            ref_a = G[l][n] * fo.chain_factor(Vd, code, scales, sg, beta) + (lam_r / Vd.size) * (4.0 - 8.0 * Vd)
            g = host(grads[(l, n)]).astype(np.float64)
            ea, eb = rel_l2(g, ref_a), rel_l2(g, dV_o[l][n])
            worst_a, worst_b = max(worst_a, ea), max(worst_b, eb)
            assert ea <= 4e-2, (l, n, ea)
            assert eb <= 0.25, (l, n, eb)
            big = np.abs(dV_o[l][n]) > 0.3 * np.abs(dV_o[l][n]).max()
            assert np.mean(np.sign(g[big]) == np.sign(dV_o[l][n][big])) >= 0.97, (l, n)
    print("worst relative dV error over the 14 linears: backward alone %.3g, whole step %.3g" % (worst_a, worst_b))
    # ---- state after the update: Adam's first step is lr * sign-like; V stays in [0, 1]
    for l in range(cfg["n_layers"]):
        for n in so.LINEARS:
            V0 = state[l][n][0]
            Vn = host(model.lin[l][n].V)
            assert Vn.min() >= 0.0 and Vn.max() <= 1.0
            assert np.max(np.abs(Vn - V0)) <= lr * 1.001 + 1e-7
            moved = np.abs(dV_o[l][n]) > 0.3 * np.abs(dV_o[l][n]).max()
            assert np.mean(np.sign(V0 - Vn)[moved] == np.sign(dV_o[l][n])[moved]) >= 0.97


def test_stage2_steps_reduce_the_alignment_loss(ctx):
    cfg, ocfg, params, W_fp, state, tokens = small_model(1)
    B, S = tokens.shape
    dparams = {k: (dev_bf16(v) if k in ("embed", "lm_head") else dev_f32(v)) for k, v in params.items()}
    dweights = [{n: dev_bf16(W_fp[l][n]) for n in so.LINEARS} for l in range(cfg["n_layers"])]
    model = stage2.Stage2Model(ctx, stage2.ModelConfig(**cfg), dparams, dweights, B, S)
    tok = torch.from_numpy(tokens.reshape(-1).astype(np.int32)).to(DEV)
    fp = model.forward(tok, quantised=False)[:2]
    hist = []
    for t in range(30):
        model.step(tok, beta=4.0 + t * 0.5, lr=5e-3, lambda_round=0.1, fp_outputs=fp)
        hist.append(host(model.loss).copy())
    faar.check_status(ctx, model.ws)
    hist = np.array(hist)
    print("L_KL, L_MSE first -> last:", hist[0], hist[-1])
    assert hist[-1, 1] < 0.8 * hist[0, 1] and hist[-1, 0] < hist[0, 0]
    packed = model.harden()
    for l in range(cfg["n_layers"]):
        for n in so.LINEARS:
            lin = model.lin[l][n]
            p_o, _, _ = fo.harden_pack(host(lin.V), host(lin.code), host(lin.scales), host(lin.s_global)[0])
            assert np.array_equal(host(packed[l][n]), p_o)


@pytest.mark.parametrize("hidden,heads,kv_heads,ffn,layers", [
    (128, 2, 1, 256, 5),          # four blocks in one launch, then one
    (2048, 32, 8, 2048, 1)])      # a block above the limit: group by group
def test_soft_weights_of_a_model_are_those_of_its_linears(ctx, hidden, heads, kv_heads, ffn, layers):
    """The forward pass forms the BF16 soft weights of many linears per launch: bit for bit what each linear's own
    evaluation gives."""
    gen = torch.Generator(device=DEV).manual_seed(3)
    cfg = stage2.ModelConfig(vocab=64, hidden=hidden, n_layers=layers, n_heads=heads, n_kv_heads=kv_heads, head_dim=64, ffn=ffn)
    rand = lambda *s: (0.05 * torch.randn(s, device=DEV, generator=gen)).to(torch.bfloat16)
    params = {"embed": rand(64, hidden), "lm_head": rand(64, hidden), "final_norm": torch.ones(hidden, device=DEV)}
    for l in range(layers):
        params[f"attn_norm.{l}"] = params[f"mlp_norm.{l}"] = torch.ones(hidden, device=DEV)
    weights = [{n: rand(*s) for n, s in cfg.linear_shapes().items()} for _ in range(layers)]
    model = stage2.Stage2Model(ctx, cfg, params, weights, 1, 16)
    for lins in model.lin:
        for x in lins.values():
            x.V.uniform_(0, 1, generator=gen)
    model.forward(torch.arange(16, dtype=torch.int32, device=DEV), quantised=True, beta=5.0)
    for lins in model.lin:
        for x in lins.values():
            alone = torch.empty_like(x.Wsoft)
            faar.softquant_eval(ctx, faar.make_shape(x.O, x.K, 16), x.V, x.code, x.scales, x.s_global, 5.0, None, None, alone)
            assert torch.equal(x.Wsoft, alone)


def test_both_forward_passes_at_once_give_the_same_step(ctx):
    """The frozen pass on the context's side stream next to the quantised one: losses and every V bit for bit those of one
    pass after the other, over several steps enqueued without a synchronisation, also on a stream of the caller's."""
    cfg, _, params, W_fp, _, tokens = small_model(1)
    B, S = tokens.shape
    dparams = {k: (dev_bf16(v) if k in ("embed", "lm_head") else dev_f32(v)) for k, v in params.items()}
    dweights = [{n: dev_bf16(W_fp[l][n]) for n in so.LINEARS} for l in range(cfg["n_layers"])]
    tok = torch.from_numpy(tokens.reshape(-1).astype(np.int32)).to(DEV)
    own = torch.cuda.Stream()
    runs = []
    try:
        for stream, overlap in ((torch.cuda.current_stream(), False), (torch.cuda.current_stream(), True), (own, True)):
            torch.cuda.synchronize()
            ctx.set_stream(stream)
            with torch.cuda.stream(stream):
                model = stage2.Stage2Model(ctx, stage2.ModelConfig(**cfg), dparams, dweights, B, S)
                assert model.overlap
                model.overlap = overlap
                losses = []
                for _ in range(4):
                    model.step(tok, beta=4.0)
                    losses.append(model.loss.clone())
                torch.cuda.synchronize()
                faar.check_status(ctx, model.ws)
                runs.append(losses + [x.V for lins in model.lin for x in lins.values()])
    finally:
        torch.cuda.synchronize()
        ctx.set_stream(torch.cuda.current_stream())
    for other in runs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(runs[0], other))


def test_stage2_step_with_a_split_lm_head_gradient_matches_the_oracle(ctx, monkeypatch):
    """A vocabulary long enough for the last hidden state's gradient, which contracts over it, to be split over CTA pairs: a
    product of the same sizes, on which alone the choice depends, says so."""
    T, hidden, vocab = 2 * 96, 128, 1600
    shape = faar.make_shape(vocab, hidden, T)
    ws = torch.empty(faar.workspace_size(shape), dtype=torch.uint8, device=DEV)
    faar.workspace_init(ctx, ws)
    dY, Ws, dX = (torch.zeros(s, dtype=torch.bfloat16, device=DEV) for s in ((T, vocab), (vocab, hidden), (T, hidden)))
    faar.layer_dx_operand(ctx, shape, dY, Ws, dX, ws)
    bn, pairs = faar.last_gemm_config(ctx)[:2]
    assert (bn, pairs) == (64, 4 * 2)
    build = small_model
    monkeypatch.setitem(globals(), "small_model", lambda seed=0: build(seed, vocab=1600))
    test_stage2_step_matches_the_oracle(ctx)


def test_a_changed_configuration_counts_from_the_next_pass_on(ctx):
    cfg, _, params, W_fp, _, tokens = small_model(1)
    B, S = tokens.shape
    dparams = {k: (dev_bf16(v) if k in ("embed", "lm_head") else dev_f32(v)) for k, v in params.items()}
    dweights = [{n: dev_bf16(W_fp[l][n]) for n in so.LINEARS} for l in range(cfg["n_layers"])]
    tok = torch.from_numpy(tokens.reshape(-1).astype(np.int32)).to(DEV)
    new = lambda **kw: stage2.Stage2Model(ctx, stage2.ModelConfig(**cfg, **kw), dparams, dweights, B, S)
    model, want = new(), new(eps=0.5, theta=100.0)
    before = model.forward(tok, quantised=True)[0]
    model.cfg.eps, model.cfg.theta = 0.5, 100.0
    after = model.forward(tok, quantised=True)[0]
    assert torch.equal(after, want.forward(tok, quantised=True)[0]) and not torch.equal(after, before)


def test_gradients_of_a_step_that_failed_are_not_written_later(ctx, monkeypatch):
    """A step that wanted dV and ran out of memory between its allocations leaves no address of a freed gradient behind."""
    cfg, _, params, W_fp, _, tokens = small_model(1)
    B, S = tokens.shape
    dparams = {k: (dev_bf16(v) if k in ("embed", "lm_head") else dev_f32(v)) for k, v in params.items()}
    dweights = [{n: dev_bf16(W_fp[l][n]) for n in so.LINEARS} for l in range(cfg["n_layers"])]
    model = stage2.Stage2Model(ctx, stage2.ModelConfig(**cfg), dparams, dweights, B, S)
    tok = torch.from_numpy(tokens.reshape(-1).astype(np.int32)).to(DEV)
    held = lambda: [getattr(b, g).lin[i].dV for b in model._blocks for g in ("qkv", "o", "gate_up", "down") for i in range(3)]
    assert len(model.step(tok, beta=4.0, want_dv=True)["dV"]) == 7 * cfg["n_layers"] and not any(held())
    real, left = torch.empty, [0]

    def empty(size, *a, **kw):
        if kw.get("dtype") == torch.float32 and len(size) == 2:              # a gradient
            left[0] -= 1
            if left[0] < 0:
                raise torch.cuda.OutOfMemoryError("no room")
        return real(size, *a, **kw)

    for n in (0, 5):
        left[0] = n
        with monkeypatch.context() as m:
            m.setattr(stage2.torch, "empty", empty)
            with pytest.raises(torch.cuda.OutOfMemoryError):
                model.step(tok, beta=4.0, want_dv=True)
        assert not any(held())
    with pytest.raises(faar.FaarError):                                      # refused by the call itself
        model.backward(torch.zeros((B * S, 8), dtype=torch.bfloat16, device=DEV), model.pos, real(256, dtype=torch.uint8, device=DEV),
                       faar.make_hparams(beta=4.0, step=1), want_dv=True)
    assert not any(held())
    torch.cuda.synchronize()


def test_the_passes_of_a_model_refuse_what_their_kernels_cannot_take(ctx):
    """Every refusal comes from a comparison on the host: nothing is launched."""
    cfg, _, params, W_fp, _, tokens = small_model(2)
    B, S = tokens.shape
    dparams = {k: (dev_bf16(v) if k in ("embed", "lm_head") else dev_f32(v)) for k, v in params.items()}
    dweights = [{n: dev_bf16(W_fp[l][n]) for n in so.LINEARS} for l in range(cfg["n_layers"])]
    model = stage2.Stage2Model(ctx, stage2.ModelConfig(**cfg), dparams, dweights, B, S)
    T, tok = B * S, torch.from_numpy(tokens.reshape(-1).astype(np.int32)).to(DEV)
    arenas = {k: torch.empty(n, dtype=torch.uint8, device=DEV) for k, n in model.arena_bytes.items()}
    scratch = torch.empty(model.scratch_bytes, dtype=torch.uint8, device=DEV)
    Z, dZ = (torch.zeros((T, cfg["vocab"]), dtype=torch.bfloat16, device=DEV) for _ in range(2))
    H, dH = (torch.zeros((T, cfg["hidden"]), dtype=torch.bfloat16, device=DEV) for _ in range(2))
    hp = faar.make_hparams(beta=4.0, step=1)

    def refused(status, calls="fqbp", block=None, beta=4.0, shape=(B, S), arena=None, **fields):
        m = faar.Model.from_buffer_copy(model._table())
        blocks = (faar.Block * cfg["n_layers"]).from_buffer_copy(model._blocks)
        for k, v in fields.items():
            setattr(m, k, v(getattr(m, k)) if callable(v) else v)
        if block:
            block(blocks[1])
        m.blocks = stage2.ctypes.addressof(blocks)
        big, small = arena if arena is not None else (arenas[True], arenas[False])
        run = {"f": lambda: faar.model_forward(ctx, m, *shape, tok, model.pos, 0, beta, 0, small, Z, H, model.ws),
               "q": lambda: faar.model_forward(ctx, m, *shape, tok, model.pos, 1, beta, 1, big, Z, H, model.ws),
               "p": lambda: faar.model_forward_both(ctx, m, *shape, tok, model.pos, beta, small, Z, H, big, Z, H, model.ws),
               "b": lambda: faar.model_backward(ctx, m, *shape, model.pos, hp, big, dZ, cfg["vocab"], dH, scratch, model.ws),
               "s": lambda: faar.model_sizes(m, *shape, 1), "o": lambda: faar.model_overlap(m, *shape)}
        for c in calls:
            with pytest.raises(faar.FaarError) as e:
                run[c]()
            assert e.value.status == status, (c, fields, e.value.status)

    off = lambda n: lambda p: p + n
    for name, n in (("embed", 2), ("lm_head", 8), ("final_norm", 4)):
        refused(faar.ERR_ALIGN, **{name: off(n)})
        refused(faar.ERR_INVALID_ARG, **{name: None})
    refused(faar.ERR_ALIGN, "b", lm_head_t=off(2))
    refused(faar.ERR_INVALID_ARG, "b", lm_head_t=None)
    for eps in (-1e-5, float("nan"), float("inf")):
        refused(faar.ERR_INVALID_ARG, eps=eps)
    for theta in (1.0, 0.5, float("nan"), float("inf")):
        refused(faar.ERR_INVALID_ARG, theta=theta)
    for beta in (0.0, float("nan"), float("inf")):
        refused(faar.ERR_INVALID_ARG, "qp", beta=beta)
    for field in ("attn_norm", "mlp_norm"):
        refused(faar.ERR_ALIGN, block=lambda b: setattr(b, field, getattr(b, field) + 4))
        refused(faar.ERR_INVALID_ARG, block=lambda b: setattr(b, field, None))
    refused(faar.ERR_ALIGN, "f", block=lambda b: setattr(b.o, "W", b.o.W + 2))
    refused(faar.ERR_ALIGN, "qbp", block=lambda b: setattr(b.o, "Wsoft", b.o.Wsoft + 2))
    refused(faar.ERR_ALIGN, "qbp", block=lambda b: setattr(b.qkv.lin[2], "V", b.qkv.lin[2].V + 4))
    refused(faar.ERR_ALIGN, "qbp", block=lambda b: setattr(b.down.lin[0], "code", b.down.lin[0].code + 1))
    refused(faar.ERR_INVALID_ARG, "qbp", block=lambda b: setattr(b.down.lin[0], "scales", None))
    refused(faar.ERR_INVALID_ARG, "b", block=lambda b: setattr(b.gate_up.lin[1], "adam_u", None))
    refused(faar.ERR_INVALID_ARG, block=lambda b: setattr(b.gate_up, "n", 1))
    refused(faar.ERR_SHAPE, block=lambda b: setattr(b.gate_up.lin[0], "rows", 240))
    refused(faar.ERR_SHAPE, "fqbpso", shape=(0, S))
    refused(faar.ERR_SHAPE, shape=(65536, 65536))
    refused(faar.ERR_SHAPE, "fqbpso", n_heads=1 << 25)
    refused(faar.ERR_SHAPE, "fqbpso", hidden=1 << 29)
    refused(faar.ERR_SHAPE, head_dim=32)
    refused(faar.ERR_SHAPE, vocab=cfg["vocab"] + 8)
    refused(faar.ERR_WORKSPACE, arena=(arenas[True][:-256], arenas[False][:-256]))
    refused(faar.ERR_ALIGN, arena=(arenas[True][16:], arenas[False][16:]))
    torch.cuda.synchronize()
    faar.check_status(ctx, model.ws)
