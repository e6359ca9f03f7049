"""Plain and forward products at the edges of tiles and of 16-column chunks, for every tile width and layout of the result's
rows, with nothing written beyond a row's values."""
import pytest
import torch

from paper_2603_22370_b200 import faar
from tests.gpu_helpers import DEV

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return faar.Context(0)


def _rand(seed, *shape):
    return torch.randn(shape, device=DEV, generator=torch.Generator(device=DEV).manual_seed(seed)).to(torch.bfloat16)


@pytest.mark.parametrize("width", [0, 128, 256, 512])
@pytest.mark.parametrize("transposed", [False, True])
@pytest.mark.parametrize("O,T,pad", [(256, 256, 0), (264, 129, 8), (65, 300, 7), (1000, 777, 8), (200, 1300, 0), (4096, 130, 16), (2056, 2000, 24)])
def test_plain_product_at_the_edges_of_tiles(ctx, O, T, pad, transposed, width):
    """FP32 sums of K products of magnitude |x w|, rounded to BF16."""
    K = 80
    X, W = _rand(1, T, K), _rand(2, O, K)
    rows, cols = (O, T) if transposed else (T, O)
    ld = (cols + 15) // 16 * 16 + pad // 8 * 8 if transposed else cols + pad
    shape = faar.make_shape(O, K, T, ldy=ld, yref_transposed=int(transposed))
    ws = ctx.workspace(shape)
    Y = torch.full((rows, ld), 7.0, dtype=torch.bfloat16, device=DEV)
    try:
        if width == 512:
            faar.tune_wide_tiles(ctx, 1)
        faar.tune_tile_n(ctx, min(width, 256))
        faar.layer_ref(ctx, shape, X, W, Y, ws)
        taken = faar.last_gemm_config(ctx)[0]
    finally:
        faar.tune_tile_n(ctx, 0)
        faar.tune_wide_tiles(ctx, -1)
    faar.check_status(ctx, ws)
    assert width == 0 or taken == (512 if width == 512 and max(O, T) > 256 else min(width, 256))
    ref, mag = X.double() @ W.double().T, X.double().abs() @ W.double().abs().T
    if transposed:
        ref, mag = ref.T, mag.T
    assert torch.all((Y[:, :cols].double() - ref).abs() <= K * 2.0 ** -24 * mag + 2.0 ** -8 * ref.abs())
    written = (cols + 15) // 16 * 16 if transposed else cols        # a transposed row is padded with zeros to 16
    assert torch.all(Y[:, cols:written] == 0.0) and torch.all(Y[:, written:] == 7.0)


@pytest.mark.parametrize("T", [2300, 2317])                                # whole and cut last chunks of 16 rows
@pytest.mark.parametrize("K", [1472, 1488, 1536])                           # 23 k blocks; 24, the last one ragged; 24
@pytest.mark.parametrize("yref_dtype", [faar.BF16, faar.F32])
def test_plain_product_with_unaligned_rows_over_several_waves(ctx, T, K, yref_dtype):
    """99 to 110 tiles, more than there are pairs: a pair's tiles but its last store their chunks' rows one by one from 24 k blocks on."""
    O, pad = 2603, 2
    X, W = _rand(6, T, K), _rand(7, O, K)
    shape = faar.make_shape(O, K, T, ldy=O + pad, yref_dtype=yref_dtype)
    ws = ctx.workspace(shape)
    Y = torch.full((T, O + pad), 7.0, dtype=torch.bfloat16 if yref_dtype == faar.BF16 else torch.float32, device=DEV)
    faar.layer_ref(ctx, shape, X, W, Y, ws)
    assert faar.last_gemm_config(ctx)[:2] == (256, 74)
    faar.check_status(ctx, ws)
    ref, mag = X.double() @ W.double().T, X.double().abs() @ W.double().abs().T
    eps = 2.0 ** -8 if yref_dtype == faar.BF16 else 0.0
    assert torch.all((Y[:, :O].double() - ref).abs() <= K * 2.0 ** -24 * mag + eps * ref.abs())
    assert torch.all(Y[:, O:] == 7.0)


@pytest.mark.parametrize("target", ["transposed", "transposed f32", "rows"])
@pytest.mark.parametrize("O,K,T,width", [(256, 96, 256, 256), (300, 96, 200, 128), (300, 96, 1030, 256), (100, 96, 1040, 512), (600, 96, 3000, 512),
                                         # tiles of 288, 304 and 464 columns for a transposed BF16 target, of 256 otherwise
                                         (2048, 8192, 2400, 0), (2048, 8192, 2600, 0), (2000, 8192, 4090, 0)])
def test_forward_product_at_the_edges_of_tiles(ctx, O, K, T, width, target):
    """dY = 2 (Y_q - Y_ref) in BF16, Y_q in FP32 from the soft weights' BF16 operand; nothing beyond a row's T values."""
    f32, trans = target.endswith("f32"), target.startswith("transposed")
    shape = faar.make_shape(O, K, T, yref_dtype=faar.F32 if f32 else faar.BF16, yref_transposed=int(trans))
    ws = ctx.workspace(shape)
    X, W = _rand(3, T, K), (0.02 * _rand(4, O, K).float()).to(torch.bfloat16)
    scales, code = torch.empty((O, K // 16), dtype=torch.uint8, device=DEV), torch.empty((O, K // 2), dtype=torch.uint8, device=DEV)
    s_global, V = torch.empty(1, dtype=torch.float32, device=DEV), torch.empty((O, K), dtype=torch.float32, device=DEV)
    faar.softquant_init(ctx, shape, W, 0.0, scales, s_global, code, V, ws)
    Wb = torch.empty((O, K), dtype=torch.bfloat16, device=DEV)
    faar.softquant_eval(ctx, shape, V, code, scales, s_global, 6.0, None, None, Wb)
    Yref = _rand(5, O, shape.ldy) if trans else _rand(5, T, shape.ldy)
    Yref = Yref.float() if f32 else Yref
    ldt = (T + 7) // 8 * 8
    dYt, loss = torch.full((O, ldt), 7.0, dtype=torch.bfloat16, device=DEV), torch.zeros(1, device=DEV)
    try:
        if width == 512:
            faar.tune_wide_tiles(ctx, 1)
        faar.tune_tile_n(ctx, min(width, 256))
        faar.layer_fwd(ctx, shape, faar.make_hparams(beta=6.0), X, Yref, V, code, scales, s_global, dYt, loss, None, ws)
        taken = faar.last_gemm_config(ctx)
    finally:
        faar.tune_tile_n(ctx, 0)
        faar.tune_wide_tiles(ctx, -1)
    faar.check_status(ctx, ws)
    # one wave of 9 x 8 fitted tiles on a whole B200
    assert taken == ((512, 72) if target == "transposed" else (256, 74)) if width == 0 else taken[0] == width
    r = Wb.double() @ X.double().T - (Yref[:, :T] if trans else Yref[:, :O].T).double()
    err = K * 2.0 ** -24 * (Wb.double().abs() @ X.double().abs().T) + 2.0 ** -23 * r.abs()
    assert torch.all((dYt[:, :T].double() - 2.0 * r).abs() <= 2.0 * err + 2.0 ** -8 * (2.0 * r).abs())
    assert torch.all(dYt[:, T:] == 7.0)
    assert abs(loss.item() - (r * r).sum().item()) <= 1e-4 * (r * r).sum().item()
