"""Stage-2 driver: full-model alignment (Eq. 6, Procedure steps 15-24) of a Llama-style decoder model whose
linears all carry their own rounding tensor V.  Buffer management only: every arithmetic step -- embedding, norms, rotary
embedding, attention, the gated MLP, every matrix product, the loss with its gradients, the chain rule into V, the
optimiser update -- is done by the CUDA library, whose faar_model_forward / faar_model_backward enqueue a whole pass.

One step (`Stage2Model.step`):
  frozen model forward (BF16 weights)                      -> Z_fp, H_fp            Procedure 16
  quantised model forward (Eq. 2 soft weights of every V)  -> Z_q, H_q, activations Procedure 17
  faar_align_loss                                          -> L_KL, L_MSE, dZ_q, dH_q   Procedure 18-20, Eq. 6
  backward through the quantised model; per group of linears with a common input: input gradient dX = dY W_soft on the
  forward pass's soft weights, i.e. at the pre-update V, then dW GEMM + chain rule + Round Loss gradient + optimiser
  update + clip
                                                                                     Procedure 21-23
Embedding, norms and LM head are frozen and stay in BF16 / FP32; the seven linears of every block are quantised.
"""
from __future__ import annotations

import ctypes
import operator
from dataclasses import dataclass

import torch

from . import faar

LINEARS = ("q_proj", "k_proj", "v_proj", "o_proj", "gate_proj", "up_proj", "down_proj")
GROUPS = {"qkv": ("q_proj", "k_proj", "v_proj"), "gate_up": ("gate_proj", "up_proj")}      # linears with a common input


@dataclass
class ModelConfig:
    vocab: int
    hidden: int
    n_layers: int
    n_heads: int
    n_kv_heads: int
    head_dim: int
    ffn: int
    eps: float = 1e-5
    theta: float = 10000.0

    def linear_shapes(self) -> dict:
        d, q, kv, f = self.hidden, self.n_heads * self.head_dim, self.n_kv_heads * self.head_dim, self.ffn
        return {"q_proj": (q, d), "k_proj": (kv, d), "v_proj": (kv, d), "o_proj": (d, q),
                "gate_proj": (f, d), "up_proj": (f, d), "down_proj": (d, f)}


class QuantLinear:
    """Device state of one quantised linear: frozen W, its NVFP4 bracket (scales, code, tensor scale), the
    rounding tensor V with its Adam moments, and a BF16 buffer for the soft weights of the current step."""

    def __init__(self, ctx: faar.Context, W: torch.Tensor, ws: torch.Tensor, opt: int = 1, Wsoft: torch.Tensor | None = None):
        O, K = W.shape
        dev = W.device
        self.W, self.O, self.K = W, O, K
        self.scales = torch.empty((O, K // 16), dtype=torch.uint8, device=dev)
        self.code = torch.empty((O, K // 2), dtype=torch.uint8, device=dev)
        self.s_global = torch.empty(1, dtype=torch.float32, device=dev)
        self.V = torch.empty((O, K), dtype=torch.float32, device=dev)
        self.m = torch.zeros((O, K), dtype=torch.float32, device=dev) if opt == 1 else None
        self.u = torch.zeros((O, K), dtype=torch.float32, device=dev) if opt == 1 else None
        self.Wsoft = Wsoft if Wsoft is not None else torch.empty((O, K), dtype=torch.bfloat16, device=dev)
        faar.softquant_init(ctx, faar.make_shape(O, K, 8), W, 0.0, self.scales, self.s_global, self.code, self.V, ws)


class Stage2Model:
    """A decoder model on one GPU.  params: "embed" [vocab, hidden] bf16, "lm_head" [vocab, hidden] bf16,
    "final_norm", "attn_norm.l", "mlp_norm.l" [hidden] float32; weights[l][name]: [O, K] bf16 (frozen)."""

    def __init__(self, ctx: faar.Context, cfg: ModelConfig, params: dict, weights: list, batch: int, seq: int, opt: int = 1):
        self.ctx, self.cfg, self.params, self.opt = ctx, cfg, params, opt
        self.batch, self.seq, self.T = batch, seq, batch * seq
        assert cfg.vocab % 16 == 0 and cfg.hidden % 16 == 0 and cfg.ffn % 16 == 0 and cfg.head_dim in (64, 128)
        dev = params["embed"].device
        self.dev = dev
        T, c = self.T, cfg
        shapes = c.linear_shapes()
        # q / k / v read the same input, and so do gate / up: each group is one matrix product over the stacked
        # weights (forward) and one input-gradient product over the stacked output gradients (backward)
        self.group_rows = {g: [shapes[n][0] for n in names] for g, names in GROUPS.items()}
        ws_shapes = list(shapes.values()) + [(sum(self.group_rows[g]), shapes[names[0]][1]) for g, names in GROUPS.items()]
        self.ws = torch.empty(max(faar.workspace_size(faar.make_shape(o, k, T)) for o, k in ws_shapes), dtype=torch.uint8,
                              device=dev)
        faar.workspace_init(ctx, self.ws)
        self.lin, self.w_group, self.wsoft_group = [], [], []
        for l in range(c.n_layers):
            lins, wg, wsg = {}, {}, {}
            for g, names in GROUPS.items():
                wg[g] = torch.cat([weights[l][n] for n in names], dim=0).contiguous()
                wsg[g] = torch.empty_like(wg[g])
                r0 = 0
                for n in names:
                    r1 = r0 + shapes[n][0]
                    lins[n] = QuantLinear(ctx, wg[g][r0:r1], self.ws, opt, Wsoft=wsg[g][r0:r1])
                    r0 = r1
            for n in LINEARS:
                if n not in lins:
                    lins[n] = QuantLinear(ctx, weights[l][n], self.ws, opt)
            self.lin.append(lins)
            self.w_group.append(wg)
            self.wsoft_group.append(wsg)
        self.pos = torch.arange(seq, dtype=torch.int32, device=dev).repeat(batch)
        self.lm_head_t = torch.empty((c.hidden, (c.vocab + 7) // 8 * 8), dtype=torch.bfloat16, device=dev)
        faar.transpose_bf16(ctx, c.vocab, c.hidden, params["lm_head"], c.hidden, self.lm_head_t, self.lm_head_t.shape[1])
        self.aws = torch.empty(faar.align_loss_workspace_size(T, c.vocab), dtype=torch.uint8, device=dev)
        faar.workspace_init(ctx, self.aws)
        self.loss = torch.zeros(2, dtype=torch.float32, device=dev)
        self.step_count = 0
        self._held, self._model, self._blocks = None, None, None
        table = self._table()
        self.arena_bytes = {bool(k): faar.model_sizes(table, batch, seq, k)[0] for k in (0, 1)}
        self.scratch_bytes = faar.model_sizes(table, batch, seq, 1)[1]
        self.overlap = faar.model_overlap(table, batch, seq)
        self._regions, self._regions_of = None, None

    # ---- helpers ------------------------------------------------------------------------------------
    def _new(self, cols, dtype=torch.bfloat16):
        return torch.empty((self.T, cols), dtype=dtype, device=self.dev)

    def _stats_bytes(self) -> int:
        """Bytes of the statistics that a pass's logits leave for the loss, 0 where a step is faster without."""
        T, vocab = self.T, self.cfg.vocab
        return faar.logit_stats_size(self.ctx, T, vocab) if faar.logit_stats_pay(self.ctx, T, vocab) else 0

    def _plan_regions(self):
        """Where the buffers of a small model's step lie in its one allocation: (name, first byte, bytes)."""
        z, h = 2 * self.T * self.cfg.vocab, 2 * self.T * self.cfg.hidden
        stats = self._stats_bytes()
        self._regions, at = [], 0
        for name, n in (("fp", self.arena_bytes[False]), ("q", self.arena_bytes[True]), ("scratch", self.scratch_bytes), ("Z_fp", z),
                        ("H_fp", h), ("Z_q", z), ("H_q", h), ("dZ", z), ("dH", h), ("stats_fp", stats), ("stats_q", stats)):
            self._regions.append((name, at, n))
            at += (n + 255) // 256 * 256
        self._region_bytes, self._regions_of = at, (self.cfg.vocab, self.cfg.hidden)

    def _groups(self, l):
        """(field, names, frozen weights, soft weights) of a block's groups of linears with a common input."""
        lin, wg, wsg = self.lin[l], self.w_group[l], self.wsoft_group[l]
        return (("qkv", GROUPS["qkv"], wg["qkv"], wsg["qkv"]), ("o", ("o_proj",), lin["o_proj"].W, lin["o_proj"].Wsoft),
                ("gate_up", GROUPS["gate_up"], wg["gate_up"], wsg["gate_up"]),
                ("down", ("down_proj",), lin["down_proj"].W, lin["down_proj"].Wsoft))

    _STATE = operator.attrgetter("W", "Wsoft", "V", "code", "scales", "s_global", "m", "u")

    def _table(self) -> faar.Model:
        """The model as the library takes it: the configuration's values and the addresses of the tensors that the attributes
        hold now, read on every call (the structure is only rebuilt if one of them has changed)."""
        p, c = self.params, self.cfg
        held = [p["embed"], p["lm_head"], p["final_norm"], self.lm_head_t]
        for l, lins in enumerate(self.lin):
            held += (p[f"attn_norm.{l}"], p[f"mlp_norm.{l}"], *self.w_group[l].values(), *self.wsoft_group[l].values())
            for x in lins.values():
                held += self._STATE(x)
        now = [c.vocab, c.hidden, c.n_layers, c.n_heads, c.n_kv_heads, c.head_dim, c.ffn, c.eps, c.theta]
        now += [0 if t is None else t.data_ptr() for t in held]
        if now == self._held:
            return self._model
        assert all(t is None or t.is_cuda for t in held), "device tensors only"
        ptr = lambda t: None if t is None else t.data_ptr()
        blocks = (faar.Block * c.n_layers)()
        for l in range(c.n_layers):
            for field, names, W, Wsoft in self._groups(l):
                g = getattr(blocks[l], field)
                g.n, g.W, g.Wsoft = len(names), ptr(W), ptr(Wsoft)
                for i, n in enumerate(names):
                    x = self.lin[l][n]
                    g.lin[i] = faar.Linear(x.O, ptr(x.V), ptr(x.code), ptr(x.scales), ptr(x.s_global), ptr(x.m), ptr(x.u), None)
            blocks[l].attn_norm, blocks[l].mlp_norm = ptr(p[f"attn_norm.{l}"]), ptr(p[f"mlp_norm.{l}"])
        self._blocks, self._held = blocks, now
        self._model = faar.Model(c.vocab, c.hidden, c.n_layers, c.n_heads, c.n_kv_heads, c.head_dim, c.ffn, c.eps, c.theta,
                                 ptr(p["embed"]), ptr(p["lm_head"]), ptr(self.lm_head_t), self.lm_head_t.shape[1],
                                 ptr(p["final_norm"]), ctypes.addressof(blocks))
        return self._model

    # ---- forward -------------------------------------------------------------------------------------
    def forward(self, tokens: torch.Tensor, quantised: bool, beta: float = 4.0, keep: bool = False):
        """tokens: [batch*seq] int32 on the device.  Returns (Z [T, vocab], H [T, hidden], activations or None)."""
        return self._forward(self._table(), tokens, quantised, beta, keep)

    def _forward(self, model: faar.Model, tokens, quantised, beta=4.0, keep=False, tau=1.0, stats=None):
        arena = torch.empty(self.arena_bytes[bool(keep)], dtype=torch.uint8, device=self.dev)
        Z, H = self._new(self.cfg.vocab), self._new(self.cfg.hidden)
        args = (self.ctx, model, self.batch, self.seq, tokens, self.pos, quantised, beta, keep, arena, Z, H)
        if stats is None:
            faar.model_forward(*args, self.ws)
        else:
            faar.model_forward_stats(*args, tau, stats, self.ws)
        return Z, H, (arena if keep else None)

    def _forward_both(self, model: faar.Model, tokens, beta, tau=1.0, stats=None):
        fp, q = (torch.empty(self.arena_bytes[k], dtype=torch.uint8, device=self.dev) for k in (False, True))
        Z_fp, H_fp, Z, H = self._new(self.cfg.vocab), self._new(self.cfg.hidden), self._new(self.cfg.vocab), self._new(self.cfg.hidden)
        args = (self.ctx, model, self.batch, self.seq, tokens, self.pos, beta, fp, Z_fp, H_fp, q, Z, H)
        if stats is None:
            faar.model_forward_both(*args, self.ws)
        else:
            faar.model_forward_both_stats(*args, tau, *stats, self.ws)
        return Z_fp, H_fp, Z, H, q

    # ---- backward ------------------------------------------------------------------------------------
    def backward(self, dZ, dH, saved, hp, want_dv=False):
        """From the loss gradients at the logits and at the last hidden state back to every V (updated in place).
        Follows the quantised forward pass of the same step: every linear's Wsoft buffer is read as that pass left it.
        Returns {(l, name): dV} if want_dv."""
        return self._backward(self._table(), dZ, dH, saved, hp, want_dv)

    def _backward(self, model: faar.Model, dZ, dH, saved, hp, want_dv):
        grads = {}
        if want_dv:
            grads = {(l, n): torch.empty((x.O, x.K), dtype=torch.float32, device=self.dev)
                     for l, lins in enumerate(self.lin) for n, x in lins.items()}
        scratch = torch.empty(self.scratch_bytes, dtype=torch.uint8, device=self.dev)
        if not want_dv:
            faar.model_backward(self.ctx, model, self.batch, self.seq, self.pos, hp, saved, dZ, dZ.shape[1], dH, scratch, self.ws)
            return None
        # the gradients' addresses are in the structure for this call alone
        self._set_dv(grads)
        try:
            faar.model_backward(self.ctx, model, self.batch, self.seq, self.pos, hp, saved, dZ, dZ.shape[1], dH, scratch, self.ws)
        finally:
            self._set_dv({})
        return grads

    def _set_dv(self, grads):
        for l in range(self.cfg.n_layers):
            for field, names, _, _ in self._groups(l):
                for i, n in enumerate(names):
                    g = grads.get((l, n))
                    getattr(self._blocks[l], field).lin[i].dV = None if g is None else g.data_ptr()

    # ---- one step of Eq. 6 -----------------------------------------------------------------------------
    def step(self, tokens: torch.Tensor, beta: float, tau: float = 1.0, lambda_kl: float = 1.0, lambda_round: float = 1.0,
             lr: float = 5e-4, want_dv: bool = False, fp_outputs=None):
        """One alignment step on a batch of token ids ([batch*seq] int32, device).  Losses {L_KL, L_MSE} are left in
        self.loss (device).  fp_outputs = (Z_fp, H_fp) reuses a frozen-model forward of the same batch.  want_dv: also
        return the quantised model's outputs, the loss gradients and every linear's dV (for inspection)."""
        self.step_count += 1
        model = self._table()
        hp = faar.make_hparams(beta=beta, lambda_round=lambda_round, opt=self.opt, lr=lr, step=self.step_count)
        if fp_outputs is None and self.overlap and not want_dv:
            # nothing of the passes is handed out: one allocation and addresses in it instead of nine tensors
            c = self.cfg
            if self._regions_of != (c.vocab, c.hidden):
                self._plan_regions()
            memory = torch.empty(self._region_bytes, dtype=torch.uint8, device=self.dev)
            base = memory.data_ptr()
            r = {name: faar.Region(base + at, n) for name, at, n in self._regions}
            passes = (self.ctx, model, self.batch, self.seq, tokens, self.pos, beta, r["fp"], r["Z_fp"], r["H_fp"], r["q"], r["Z_q"], r["H_q"])
            loss = (self.ctx, self.T, c.vocab, c.hidden, r["Z_fp"], r["Z_q"], c.vocab, r["H_fp"], r["H_q"], c.hidden, tau, lambda_kl)
            if r["stats_q"].numel():
                faar.model_forward_both_stats(*passes, tau, r["stats_fp"], r["stats_q"], self.ws)
                faar.align_loss_stats(*loss, r["stats_fp"], r["stats_q"], r["dZ"], r["dH"], self.loss, self.aws)
            else:
                faar.model_forward_both(*passes, self.ws)
                faar.align_loss(*loss, r["dZ"], r["dH"], self.loss, self.aws)
            faar.model_backward(self.ctx, model, self.batch, self.seq, self.pos, hp, r["q"], r["dZ"], c.vocab, r["dH"], r["scratch"], self.ws)
            return None
        c, T = self.cfg, self.T
        n = self._stats_bytes()                # as above: the step is the same, bit for bit, whatever is handed in or out
        stats = tuple(torch.empty(n, dtype=torch.uint8, device=self.dev) for _ in range(2)) if n else ()
        st_fp, st_q = stats or (None, None)
        if fp_outputs is None and self.overlap:
            Z_fp, H_fp, Z_q, H_q, saved = self._forward_both(model, tokens, beta, tau, stats or None)
        else:
            if fp_outputs is None:
                Z_fp, H_fp = self._forward(model, tokens, quantised=False, tau=tau, stats=st_fp)[:2]
            else:
                Z_fp, H_fp = fp_outputs
                if n:
                    faar.logit_stats(self.ctx, T, c.vocab, Z_fp, c.vocab, tau, st_fp)
            Z_q, H_q, saved = self._forward(model, tokens, quantised=True, beta=beta, keep=True, tau=tau, stats=st_q)
        dZ, dH = torch.empty_like(Z_q), torch.empty_like(H_q)
        loss = faar.align_loss_stats if stats else faar.align_loss
        loss(self.ctx, T, c.vocab, c.hidden, Z_fp, Z_q, Z_q.shape[1], H_fp, H_q, c.hidden, tau, lambda_kl, *stats, dZ, dH, self.loss, self.aws)
        grads = self._backward(model, dZ, dH, saved, hp, want_dv)
        return {"Z_q": Z_q, "H_q": H_q, "dZ": dZ, "dH": dH, "dV": grads} if want_dv else None

    def round_loss_sum(self) -> float:
        """Sum over all linears of the Round Loss (Eq. 6's third term without lambda); reads back one float each."""
        out = torch.zeros(1, dtype=torch.float32, device=self.dev)
        total = 0.0
        for layer in self.lin:
            for lin in layer.values():
                faar.round_loss(self.ctx, lin.V, lin.O * lin.K, out, self.ws)
                total += float(out.item())
        return total

    def harden(self) -> list:
        """Eq. 7 for every linear: packed NVFP4 codes (the scales and tensor scale are the set-up's)."""
        res = []
        for layer in self.lin:
            d = {}
            for n, lin in layer.items():
                packed = torch.empty((lin.O, lin.K // 2), dtype=torch.uint8, device=self.dev)
                faar.harden_pack(self.ctx, faar.make_shape(lin.O, lin.K, 8), lin.V, lin.code, lin.scales, lin.s_global, packed,
                                 None, None, None)
                d[n] = packed
            res.append(d)
        faar.check_status(self.ctx, self.ws)
        return res
