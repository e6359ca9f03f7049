"""dW launches of short contractions (256-wide tiles, eight weights per lane and request): the same update, bit for bit, as
tiles of 128 columns, whose lanes take four weights, for rows and columns that fill no tile, the last contraction that counts
as short and the first that does not, state tensors on and off 32-byte boundaries, and every optimiser form."""
import numpy as np
import pytest
import torch

from paper_2603_22370_b200 import faar
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
            V, m, u, dV = _shifted(V0, shift), _shifted(m0, shift), _shifted(u0, shift), _shifted(torch.zeros_like(V0), shift)
            call = faar.layer_bwd_rowmajor if row_major else faar.layer_bwd
            call(ctx, shape, hp, dY, X, V, code, scales, s_global, m if adam else None, u if adam else None, dV, ws)
            assert faar.last_gemm_config(ctx)[0] == width
            torch.cuda.synchronize()
            faar.check_status(ctx, ws)
            soft = [host(ws[OPERAND:OPERAND + 2 * O * K]).copy()] if chained else []      # the next step's operand
            out.append([host(t).copy() for t in (V, m, u, dV)] + soft)
    finally:
        faar.tune_tail_split(ctx, -1)
        faar.tune_tile_n(ctx, 0)
    assert np.isfinite(out[0][0]).all() and not np.array_equal(out[0][0], host(V0))
    for a, b in zip(out[0], out[1]):
        assert np.array_equal(a, b)
