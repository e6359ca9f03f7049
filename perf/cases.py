"""What is measured: calls of this framework as its users make them, over the sizes and options that they use.

Kinds of case
  step      one optimisation step of a linear layer on a calibration batch in HBM (forward, loss, backward, update)
  host      the same step with the batch in pinned host memory, alternating between two sets of staging buffers
  run       the whole layer-wise optimisation of one linear: set-up, steps, hardening and packing
  quantise  a weight matrix to deployable NVFP4 by rounding to nearest: scales, bracket, hardening, tiled scales
  deployed  a hardened linear's product with activations that are quantised on the way in
  align     one full-model alignment step of a decoder model: both forward passes, loss, backward, every update
Activations have heavy-tailed values or outlier channels, weights a few outliers, as the package's input recipes do.
"""
import math

import torch

from paper_2603_22370_b200 import faar, stage1, stage2

DEV = "cuda:0"
#: steps of one optimisation run; the temperature of step t follows the package's schedule, then a new run begins
RUN_STEPS = 200

#: the decoder models of the alignment cases: heads of 64 and of 128 elements, and the small one of the tests
MODELS = {
    "heads64": dict(hidden=2048, n_heads=32, n_kv_heads=8, head_dim=64, ffn=8192),
    "heads128": dict(hidden=2048, n_heads=16, n_kv_heads=8, head_dim=128, ffn=6144),
    "small64": dict(hidden=128, n_heads=2, n_kv_heads=1, head_dim=64, ffn=256),
    "small128": dict(hidden=512, n_heads=4, n_kv_heads=2, head_dim=128, ffn=1024),
}


def listed():
    return [
        # the small parity layer, chained steps as the layer-wise driver takes them: launches and latency count
        dict(name="step_small_layer", kind="step", O=128, K=256, T=1024, chained=True, act_quant=False, adam=True, target_f32=False),
        # sizes that fill no tile, a row-major FP32 target and plain gradient descent: a caller with its own layout
        dict(name="step_ragged", kind="step", O=1000, K=1040, T=777, chained=False, act_quant=False, adam=False, target_f32=True),
        # gate_proj of a 1B decoder block on quantised activations, chained
        dict(name="step_gate_proj", kind="step", O=8192, K=2048, T=4096, chained=True, act_quant=True, adam=True, target_f32=False),
        # down_proj of a 1B decoder block: the headline benchmark's step
        dict(name="step_down_proj", kind="step", O=2048, K=8192, T=4096, chained=False, act_quant=False, adam=True, target_f32=False),
        # the same layer with a batch that arrives from the host every step
        dict(name="step_from_host", kind="host", O=2048, K=8192, T=1024),
        # k_proj of a 1B decoder block from its weights to its packed form, with a short schedule
        dict(name="run_k_proj", kind="run", O=512, K=2048, T=4096, steps=12, act_quant=False),
        # converting an up_proj: set-up and pack kernels alone
        dict(name="quantise_up_proj", kind="quantise", O=8192, K=2048, w_f32=False),
        # inference with a hardened down_proj on a prompt, and with a hardened gate_proj on one token per sequence
        dict(name="deployed_prefill", kind="deployed", O=2048, K=8192, T=4096),
        dict(name="deployed_decode", kind="deployed", O=8192, K=2048, T=8),
        # alignment of the tests' model on short sequences: a long chain of small launches
        dict(name="align_small_model", kind="align", model="small64", layers=2, vocab=512, batch=2, seq=96),
        # alignment of a 1B-shaped model (four of its blocks) at the benchmark's batch and vocabulary
        dict(name="align_heads64", kind="align", model="heads64", layers=4, vocab=128256, batch=4, seq=2048),
        # alignment of a model with 128-element heads on shorter sequences
        dict(name="align_heads128", kind="align", model="heads128", layers=2, vocab=32000, batch=2, seq=1000),
    ]


def _log_int(rng, lo, hi, multiple=1):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / multiple)) * multiple
    return min(max(v, lo), hi)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "run", "quantise", "deployed", "deployed", "align", "align", "host"])
    O, K, T = _log_int(rng, 64, 8192), _log_int(rng, 128, 8192, 16), _log_int(rng, 64, 4096)
    if rng.random() < 0.5:                       # most layers have round widths; batches are ragged more often
        O = (O + 63) // 64 * 64
    if O * K > 8192 * 2048:
        O = 8192 * 2048 // K
    if kind == "step":
        return dict(kind=kind, O=O, K=K, T=T, chained=rng.random() < 0.5, act_quant=rng.random() < 0.3, adam=rng.random() < 0.8,
                    target_f32=rng.random() < 0.3)
    if kind == "host":
        return dict(kind=kind, O=O, K=K, T=max(64, T // 4))
    if kind == "run":
        return dict(kind=kind, O=O, K=K, T=T, steps=rng.randint(4, 16), act_quant=rng.random() < 0.3)
    if kind == "quantise":
        return dict(kind=kind, O=O, K=K, w_f32=rng.random() < 0.3)
    if kind == "deployed":
        return dict(kind=kind, O=O, K=(K + 31) // 32 * 32, T=T if rng.random() < 0.6 else rng.randint(1, 64))
    model = rng.choice(sorted(MODELS))
    if model.startswith("small"):
        return dict(kind=kind, model=model, layers=rng.randint(1, 4), vocab=16 * rng.randint(16, 256), batch=rng.randint(1, 4),
                    seq=_log_int(rng, 16, 512))
    return dict(kind=kind, model=model, layers=rng.randint(1, 3), vocab=16 * _log_int(rng, 500, 4000), batch=rng.randint(1, 3),
                seq=_log_int(rng, 256, 2048))


# ---- inputs ------------------------------------------------------------------------------------------------------
def _normal(gen, *shape, sigma=1.0):
    return torch.randn(shape, device=DEV, generator=gen, dtype=torch.float32).mul_(sigma)


def _weights(gen, O, K):
    W = _normal(gen, O, K, sigma=0.02)
    return torch.where(torch.rand((O, K), device=DEV, generator=gen) < 1e-3, W * 10.0, W)


def _activations(gen, T, K):
    """Student-t values (4 degrees of freedom) with 16 outlier channels, BF16."""
    chi2 = -2.0 * torch.log(torch.rand((T, K), device=DEV, generator=gen).clamp_min_(1e-12) *
                            torch.rand((T, K), device=DEV, generator=gen).clamp_min_(1e-12))
    X = _normal(gen, T, K) / torch.sqrt(chi2 / 4.0)
    X[:, torch.randperm(K, device=DEV, generator=gen)[:16]] *= 20.0
    return X.to(torch.bfloat16)


def _layer_state(gen, O, K, T, act_quant=False, adam=True, target_f32=False, batch=True):
    """A linear in the middle of its set-up, by the library's own calls: bracket, V, moments, batch and frozen target."""
    s = {"ctx": faar.Context(0), "W": _weights(gen, O, K).to(torch.bfloat16), "t": 0, "O": O, "K": K, "T": T, "adam": adam}
    ctx = s["ctx"]
    ldt = (T + 7) // 8 * 8
    shape = s["shape"] = faar.make_shape(O, K, T, ldxt=ldt, yref_dtype=faar.F32 if target_f32 else faar.BF16,
                                         yref_transposed=0 if target_f32 else 1)
    ws = s["ws"] = torch.empty(faar.workspace_size(shape), dtype=torch.uint8, device=DEV)
    faar.workspace_init(ctx, ws)
    s["scales"] = torch.empty((O, K // 16), dtype=torch.uint8, device=DEV)
    s["code"] = torch.empty((O, K // 2), dtype=torch.uint8, device=DEV)
    s["s_global"] = torch.empty(1, dtype=torch.float32, device=DEV)
    s["V"] = torch.empty((O, K), dtype=torch.float32, device=DEV)
    s["m"] = torch.zeros((O, K), dtype=torch.float32, device=DEV) if adam else None
    s["u"] = torch.zeros((O, K), dtype=torch.float32, device=DEV) if adam else None
    s["loss"] = torch.zeros(2, dtype=torch.float32, device=DEV)
    s["act_scale"] = 0.0
    faar.softquant_init(ctx, shape, s["W"], 0.0, s["scales"], s["s_global"], s["code"], s["V"], ws)
    if batch:
        X = _activations(gen, T, K)
        s["Yref"] = torch.zeros((T, O) if target_f32 else (O, shape.ldy), dtype=torch.float32 if target_f32 else torch.bfloat16,
                                device=DEV)
        faar.layer_ref(ctx, shape, X, s["W"], s["Yref"], ws)
        if act_quant:
            Xq, sx = torch.empty_like(X), torch.empty(1, dtype=torch.float32, device=DEV)
            faar.act_fakequant(ctx, T, K, X, K, 0.0, Xq, K, sx, None, None, ws)
            s["act_scale"] = float(sx.item())
            X = Xq
        s["X"] = X
        s["Xt"] = torch.zeros((K, ldt), dtype=torch.bfloat16, device=DEV)
        faar.transpose_bf16(ctx, T, K, X, K, s["Xt"], ldt)
    return s


def _model_state(gen, case):
    m = MODELS[case["model"]]
    cfg = stage2.ModelConfig(vocab=case["vocab"], n_layers=case["layers"], **m)
    ones = lambda: torch.ones(cfg.hidden, dtype=torch.float32, device=DEV)  # noqa: E731
    bf = lambda *shape, sigma: _normal(gen, *shape, sigma=sigma).to(torch.bfloat16)  # noqa: E731
    params = {"embed": bf(cfg.vocab, cfg.hidden, sigma=1.0), "lm_head": bf(cfg.vocab, cfg.hidden, sigma=1.0 / math.sqrt(cfg.hidden)),
              "final_norm": ones()}
    weights = []
    for l in range(cfg.n_layers):
        params[f"attn_norm.{l}"], params[f"mlp_norm.{l}"] = ones(), ones()
        weights.append({n: bf(o, k, sigma=1.0 / math.sqrt(k)) for n, (o, k) in cfg.linear_shapes().items()})
    model = stage2.Stage2Model(faar.Context(0), cfg, params, weights, case["batch"], case["seq"])
    # alignment starts from rounding variables that the layer-wise stage has moved, and runs at its middle temperatures
    for layer in model.lin:
        for lin in layer.values():
            lin.V.add_(_normal(gen, lin.O, lin.K, sigma=0.2)).clamp_(0.0, 1.0)
    tokens = torch.randint(0, cfg.vocab, (case["batch"] * case["seq"],), dtype=torch.int32, device=DEV, generator=gen)
    return {"model": model, "tokens": tokens, "t": RUN_STEPS // 2}


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    kind = case["kind"]
    if kind == "align":
        s = _model_state(gen, case)
    elif kind == "step":
        s = _layer_state(gen, case["O"], case["K"], case["T"], case["act_quant"], case["adam"], case["target_f32"])
        s["chained"] = case["chained"]
    elif kind == "host":
        O, K, T = case["O"], case["K"], case["T"]
        s = _layer_state(gen, O, K, T, batch=False)
        s["X_host"] = _activations(gen, T, K).cpu().pin_memory()
        s["loss_host"] = torch.zeros(2, dtype=torch.float32).pin_memory()
        s["staging"] = [(torch.empty((T, K), dtype=torch.bfloat16, device=DEV),
                         torch.zeros((K, s["shape"].ldxt), dtype=torch.bfloat16, device=DEV),
                         torch.zeros((O, s["shape"].ldy), dtype=torch.bfloat16, device=DEV)) for _ in range(2)]
    elif kind == "run":
        s = {"ctx": faar.Context(0), "W": _weights(gen, case["O"], case["K"]).to(torch.bfloat16),
             "X": _activations(gen, case["T"], case["K"]), "steps": case["steps"], "act_quant": case["act_quant"]}
    elif kind == "quantise":
        O, K = case["O"], case["K"]
        W = _weights(gen, O, K)
        s = {"ctx": faar.Context(0), "W": W if case["w_f32"] else W.to(torch.bfloat16), "O": O, "K": K,
             "shape": faar.make_shape(O, K, 8, w_dtype=faar.F32 if case["w_f32"] else faar.BF16)}
        s["ws"] = torch.empty(faar.workspace_size(s["shape"]), dtype=torch.uint8, device=DEV)
        faar.workspace_init(s["ctx"], s["ws"])
        s["scales"] = torch.empty((O, K // 16), dtype=torch.uint8, device=DEV)
        s["code"] = torch.empty((O, K // 2), dtype=torch.uint8, device=DEV)
        s["packed"] = torch.empty((O, K // 2), dtype=torch.uint8, device=DEV)
        s["s_global"] = torch.empty(1, dtype=torch.float32, device=DEV)
        s["V"] = torch.empty((O, K), dtype=torch.float32, device=DEV)
        s["tiled"] = torch.empty(_tiled_bytes(O, K), dtype=torch.uint8, device=DEV)
    elif kind == "deployed":
        O, K, T = case["O"], case["K"], case["T"]
        s = _layer_state(gen, O, K, 8, batch=False)
        s["T"] = T
        s["packed"] = torch.empty((O, K // 2), dtype=torch.uint8, device=DEV)
        faar.harden_pack(s["ctx"], s["shape"], s["V"], s["code"], s["scales"], s["s_global"], s["packed"], None, None, None)
        s["tiled"] = torch.empty(_tiled_bytes(O, K), dtype=torch.uint8, device=DEV)
        faar.swizzle_scales(s["ctx"], O, K // 16, s["scales"], s["tiled"])
        for unused in ("V", "m", "u", "code", "W"):
            del s[unused]
        s["X"] = _activations(gen, T, K)
        s["Xq"] = torch.empty((T, K), dtype=torch.bfloat16, device=DEV)
        s["x_packed"] = torch.empty((T, K // 2), dtype=torch.uint8, device=DEV)
        s["x_scales"] = torch.empty((T, K // 16), dtype=torch.uint8, device=DEV)
        s["x_tiled"] = torch.empty(_tiled_bytes(T, K), dtype=torch.uint8, device=DEV)
        s["x_s_global"] = torch.empty(1, dtype=torch.float32, device=DEV)
        s["Y"] = torch.empty((T, O), dtype=torch.bfloat16, device=DEV)
    else:
        raise ValueError(kind)
    s["kind"] = kind
    return s


def _tiled_bytes(rows, K):
    return (rows + 127) // 128 * ((K // 16 + 3) // 4) * 512


# ---- one pass ----------------------------------------------------------------------------------------------------
def _hparams(s, chained):
    t = s["t"] % RUN_STEPS
    s["t"] += 1
    more = {}
    if chained:
        more = dict(wsoft_ready=int(t > 0), beta_next=stage1.beta_schedule(t + 1, RUN_STEPS) if t + 1 < RUN_STEPS else 0.0)
    return faar.make_hparams(beta=stage1.beta_schedule(t, RUN_STEPS), opt=int(s["adam"]), lr=1e-2 if s["adam"] else 1e-4, step=t + 1,
                             act_scale=s["act_scale"], **more)


def run(s):
    kind = s["kind"]
    if kind == "align":
        model, t = s["model"], s["t"] % RUN_STEPS
        s["t"] += 1
        model.step(s["tokens"], beta=stage1.beta_schedule(t, RUN_STEPS))
        return {"loss": model.loss, "V": [lin.V for layer in model.lin for lin in layer.values()]}
    if kind == "step":
        hp = _hparams(s, s["chained"])
        faar.layer_step(s["ctx"], s["shape"], hp, s["X"], s["Xt"], s["Yref"], s["V"], s["code"], s["scales"], s["s_global"], s["m"],
                        s["u"], s["loss"], s["ws"])
        return {"V": s["V"], "m": s["m"], "u": s["u"], "loss": s["loss"]}
    if kind == "host":
        X_dev, Xt_dev, Y_dev = s["staging"][s["t"] % 2]
        hp = _hparams(s, False)
        faar.layer_step_host(s["ctx"], s["shape"], hp, s["X_host"], None, s["W"], X_dev, Xt_dev, Y_dev, s["V"], s["code"],
                             s["scales"], s["s_global"], s["m"], s["u"], s["loss"], s["loss_host"], s["ws"])
        return {"V": s["V"], "m": s["m"], "u": s["u"], "loss": s["loss_host"]}
    if kind == "run":
        r = stage1.optimise_layer(s["ctx"], s["W"], s["X"], steps=s["steps"], quantise_activations=s["act_quant"])
        return {"packed": r["packed"], "scales": r["scales"], "V": r["V"], "s_global": r["s_global"], "losses": list(r["history"][-1][1:])}
    if kind == "quantise":
        faar.softquant_init(s["ctx"], s["shape"], s["W"], 0.0, s["scales"], s["s_global"], s["code"], s["V"], s["ws"])
        faar.harden_pack(s["ctx"], s["shape"], s["V"], s["code"], s["scales"], s["s_global"], s["packed"], None, None, None)
        faar.swizzle_scales(s["ctx"], s["O"], s["K"] // 16, s["scales"], s["tiled"])
        return {"V": s["V"], "code": s["code"], "packed": s["packed"], "scales": s["scales"], "tiled": s["tiled"], "s_global": s["s_global"]}
    O, K, T = s["O"], s["K"], s["T"]
    faar.act_fakequant(s["ctx"], T, K, s["X"], K, 0.0, s["Xq"], K, s["x_s_global"], s["x_packed"], s["x_scales"], s["ws"])
    faar.swizzle_scales(s["ctx"], T, K // 16, s["x_scales"], s["x_tiled"])
    faar.nvfp4_gemm(s["ctx"], T, O, K, s["x_packed"], s["x_tiled"], s["x_s_global"], s["packed"], s["tiled"], s["s_global"], s["Y"], O,
                    s["ws"])
    return {"Y": s["Y"], "Xq": s["Xq"], "x_packed": s["x_packed"], "x_scales": s["x_scales"], "x_s_global": s["x_s_global"]}


# ---- what a pass cannot do without -------------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "align":
        m = MODELS[case["model"]]
        cfg = stage2.ModelConfig(vocab=case["vocab"], n_layers=case["layers"], **m)
        T = case["batch"] * case["seq"]
        n = sum(o * k for o, k in cfg.linear_shapes().values()) * cfg.n_layers
        attn = 2.0 * case["batch"] * cfg.n_heads * case["seq"] ** 2 * cfg.head_dim * cfg.n_layers        # causal forward
        flops = 4 * 2.0 * T * n + 3 * 2.0 * T * cfg.vocab * cfg.hidden + (2 + 2.5) * attn
        # frozen weights, code, scales and s_global in; V, m, u in and out; LM head and the tokens' embedding rows in
        return {"flops": flops, "bytes": n * (2 + 0.5 + 1 / 16 + 24.0) + 2.0 * cfg.vocab * cfg.hidden + 2.0 * T * cfg.hidden + 4.0 * T}
    O, K = case["O"], case["K"]
    n = float(O * K)
    if kind == "quantise":
        return {"flops": 0.0, "bytes": n * ((4 if case["w_f32"] else 2) + 4 + 0.5 + 0.5) + 2 * n / 16}
    T = case["T"]
    if kind == "deployed":
        return {"flops": 2.0 * T * n, "bytes": T * K * (2 + 2 + 0.5 + 1 / 16) + n * (0.5 + 1 / 16) + 2.0 * T * O}
    if kind == "run":
        # every step reads and writes the state; weights and batch come in once
        return {"flops": (4.0 * case["steps"] + 2.0) * T * n,
                "bytes": n * (2 + 0.5 + 1 / 16) + 2.0 * T * K + case["steps"] * (n * (16.0 + 8.0 + 0.5 + 1 / 16) + 2.0 * T * O)}
    if kind == "host":
        return {"flops": 6.0 * T * n, "bytes": 2.0 * T * K + n * (2 + 24.0 + 0.5 + 1 / 16)}
    state = 24.0 if case["adam"] else 8.0
    return {"flops": 4.0 * T * n, "bytes": 2.0 * T * K + T * O * (4.0 if case["target_f32"] else 2.0) + n * (state + 0.5 + 1 / 16)}


#: About four times what was measured: layer steps against the same step with sums in 64 bits (rel 1.4e-3 in the first moments,
#: whose smallest entries differ by 2 rms), whole runs the same way (V 6.5e-4, one decision in 2000), products against the
#: 64-bit product of the decoded operands rounded to BF16 (1.3e-5, a BF16 unit at most), alignment steps against the same
#: steps with other attention kernels (V 3.6e-4 after two steps; the loss of a few tokens, a difference of two BF16 forward
#: passes, 3e-3).
TOLERANCE = {
    "step": {"rel": 6e-3, "max": 0.9},
    "host": {"rel": 6e-3, "max": 0.9},
    "run": {"rel": 3e-3, "max": 0.4, "differ": 4e-3},
    "quantise": "exact",
    "deployed": {"rel": 2e-4, "max": 0.03},
}


def tolerance(case):
    if case["kind"] == "align":
        return {"rel": 1.2e-2} if case["model"].startswith("small") else {"rel": 1.5e-3, "max": 0.02}
    return TOLERANCE[case["kind"]]
