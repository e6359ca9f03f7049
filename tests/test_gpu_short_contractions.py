"""dW launches of short contractions (256-wide tiles, eight weights per lane and request): the same update, bit for bit, as
tiles of 128 columns, whose lanes take four weights, for rows and columns that fill no tile, the last contraction that counts
as short and the first that does not, state tensors on and off 32-byte boundaries, every optimiser form, and several linears
in one launch."""
import numpy as np
import pytest
import torch

from paper_2603_22370_b200 import faar, stage2
from tests.gpu_helpers import DEV, host

pytestmark = pytest.mark.gpu
OPERAND = 129 * 1024                              # the soft weights' place in a workspace: after the header and the loss partials


@pytest.fixture(scope="module")
def ctx():
    return faar.Context(0)


def _shifted(t, floats):
    """A copy of `t` whose data begin `floats` FP32 values after a 256-byte boundary."""
    buf = torch.empty(t.numel() + floats, dtype=torch.float32, device=DEV)
    view = buf[floats:].view(t.shape)
    view.copy_(t)
    return view


@pytest.mark.parametrize("shift", [0, 4])
@pytest.mark.parametrize("adam,chained,row_major", [(True, False, False), (True, True, False), (False, False, True), (True, False, True),
                                                    (False, True, False)])
@pytest.mark.parametrize("O,K,T", [(8, 16, 8), (300, 1040, 77), (264, 272, 640), (520, 784, 2560), (520, 784, 2561)])
def test_short_contractions_give_the_same_step(ctx, O, K, T, adam, chained, row_major, shift):
    gen = torch.Generator(device=DEV).manual_seed(O + T)
    rnd = lambda *s: torch.randn(s, device=DEV, generator=gen)  # noqa: E731
    ldt, ldo = (T + 7) // 8 * 8, (O + 7) // 8 * 8
    shape = faar.make_shape(O, K, T, ldxt=ldt, ldy=ldo if row_major else O)
    ws = ctx.workspace(shape)
    scales, code = torch.empty((O, K // 16), dtype=torch.uint8, device=DEV), torch.empty((O, K // 2), dtype=torch.uint8, device=DEV)
    s_global, V0 = torch.empty(1, dtype=torch.float32, device=DEV), torch.empty((O, K), dtype=torch.float32, device=DEV)
    faar.softquant_init(ctx, shape, (0.02 * rnd(O, K)).to(torch.bfloat16), 0.0, scales, s_global, code, V0, ws)
    m0, u0 = 1e-3 * rnd(O, K), 1e-6 * rnd(O, K).abs()
    dY = rnd(T, ldo).to(torch.bfloat16) if row_major else rnd(O, ldt).to(torch.bfloat16)
    X = rnd(T, K).to(torch.bfloat16) if row_major else rnd(K, ldt).to(torch.bfloat16)
    if not row_major:
        dY[:, T:] = 0
        X[:, T:] = 0
    hp = faar.make_hparams(beta=6.0, step=2, opt=int(adam), lr=1e-2 if adam else 1e-5, beta_next=9.0 if chained else 0.0)
    out = []
    try:
        # forced: no split contraction, whose choice does not depend on the width
        faar.tune_tail_split(ctx, 0)
        for width in (256, 128):
            faar.tune_tile_n(ctx, width)
            ws[OPERAND:OPERAND + 2 * O * K] = 0xFF
            V, m, u, dV = _shifted(V0, shift), _shifted(m0, shift), _shifted(u0, shift), _shifted(torch.zeros_like(V0), shift)
            call = faar.layer_bwd_rowmajor if row_major else faar.layer_bwd
            call(ctx, shape, hp, dY, X, V, code, scales, s_global, m if adam else None, u if adam else None, dV, ws)
            assert faar.last_gemm_config(ctx)[0] == width
            torch.cuda.synchronize()
            faar.check_status(ctx, ws)
            out.append([host(t).copy() for t in (V, m, u, dV)])
            if chained:                                                   # the next step's operand
                want = torch.empty((O, K), dtype=torch.bfloat16, device=DEV)
                faar.softquant_eval(ctx, shape, V, code, scales, s_global, 9.0, None, None, want)
                assert torch.equal(ws[OPERAND:OPERAND + 2 * O * K], want.view(torch.uint8).view(-1))
    finally:
        faar.tune_tail_split(ctx, -1)
        faar.tune_tile_n(ctx, 0)
    assert np.isfinite(out[0][0]).all() and not np.array_equal(out[0][0], host(V0))
    for a, b in zip(out[0], out[1]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("opt", [1, 0])
def test_several_linears_in_one_short_contraction_give_the_same_step(ctx, opt):
    """q / k / v and gate / up stacked in one dW launch each (320 + 64 + 64 and 304 + 304 rows, which end inside tiles), some
    state tensors on 16-byte boundaries only: every gradient and update as with tiles of 128 columns."""
    cfg = stage2.ModelConfig(vocab=64, hidden=336, n_layers=1, n_heads=5, n_kv_heads=1, head_dim=64, ffn=304)
    batch, seq = 2, 72                                                    # three k blocks, the last one ragged
    out = []
    try:
        for width in (256, 128):
            gen = torch.Generator(device=DEV).manual_seed(7)
            rnd = lambda *s: (torch.randn(s, device=DEV, generator=gen) / s[-1] ** 0.5).to(torch.bfloat16)  # noqa: E731,B023
            ones = torch.ones(cfg.hidden, device=DEV)
            params = {"embed": rnd(64, cfg.hidden) * 18, "lm_head": rnd(64, cfg.hidden), "final_norm": ones, "attn_norm.0": ones,
                      "mlp_norm.0": ones}
            model = stage2.Stage2Model(ctx, cfg, params, [{n: rnd(*s) for n, s in cfg.linear_shapes().items()}], batch, seq, opt=opt)
            lins = model.lin[0]
            for x in lins.values():
                x.V.uniform_(0, 1, generator=gen)
            for name, field in (("k_proj", "V"), ("up_proj", "V"), ("up_proj", "m"), ("q_proj", "u")):
                if getattr(lins[name], field) is not None:
                    setattr(lins[name], field, _shifted(getattr(lins[name], field), 4))
            tokens = torch.arange(batch * seq, dtype=torch.int32, device=DEV) % 61
            faar.tune_tile_n(ctx, width)
            before = [host(x.V).copy() for x in lins.values()]
            for _ in range(2):
                grads = model.step(tokens, beta=6.0, want_dv=True)["dV"]
                assert faar.last_gemm_config(ctx)[0] == width             # the dW launch of q / k / v
            torch.cuda.synchronize()
            faar.check_status(ctx, model.ws)
            state = [host(t).copy() for x in lins.values() for t in (x.V, x.m, x.u) if t is not None]
            out.append(state + [host(g).copy() for g in grads.values()])
            assert all(np.isfinite(host(x.V)).all() and not np.array_equal(b, host(x.V)) for b, x in zip(before, lins.values()))
    finally:
        faar.tune_tile_n(ctx, 0)
    for a, b in zip(out[0], out[1]):
        assert np.array_equal(a, b)
