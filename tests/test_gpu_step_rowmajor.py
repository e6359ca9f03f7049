"""faar_layer_step_rowmajor: the step of faar_layer_step without the transposed batch, bit for bit."""
import pytest
import torch

from paper_2603_22370_b200 import faar

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


@pytest.mark.parametrize("O,K,T,opt", [
    (1, 16, 1, 1),                # the smallest
    (130, 144, 63, 0),            # one row more than half a row block, a narrow last column, one cut k block
    (256, 528, 65, 1),
    (300, 1040, 777, 0),
    (512, 2048, 1100, 1),         # split contraction
    (2500, 1040, 130, 1),         # more tiles than pairs
])
def test_step_on_the_row_major_batch_gives_the_same_bits(ctx, O, K, T, opt):
    gen = torch.Generator(device=DEV).manual_seed(3)
    W, X = ((torch.randn(s, device=DEV, generator=gen) * f).to(torch.bfloat16) for s, f in (((O, K), 0.05), ((T, K), 1.0)))
    ldt = (T + 7) // 8 * 8
    shape = faar.make_shape(O, K, T, ldxt=ldt, yref_transposed=1)
    ws = torch.empty(faar.workspace_size(shape), dtype=torch.uint8, device=DEV)
    faar.workspace_init(ctx, ws)
    Xt = torch.zeros((K, ldt), dtype=torch.bfloat16, device=DEV)
    faar.transpose_bf16(ctx, T, K, X, K, Xt, ldt)
    Yref = torch.zeros((O, shape.ldy), dtype=torch.bfloat16, device=DEV)
    faar.layer_ref(ctx, shape, X, W, Yref, ws)
    scales, code = (torch.empty((O, n), dtype=torch.uint8, device=DEV) for n in (K // 16, K // 2))
    s_global, V0 = torch.empty(1, device=DEV), torch.empty((O, K), device=DEV)
    faar.softquant_init(ctx, shape, W, 0.0, scales, s_global, code, V0, ws)
    out = []
    for row_major in (False, True):
        V, m, u, loss = V0.clone(), torch.zeros_like(V0), torch.zeros_like(V0), torch.zeros(2, device=DEV)
        for t in range(3):        # chained: the last two steps take the soft weights that the dW launch before left
            hp = faar.make_hparams(beta=5.0, opt=opt, lr=1e-2, step=t + 1, wsoft_ready=int(t > 0), beta_next=5.0 if t < 2 else 0.0)
            state = (Yref, V, code, scales, s_global, m, u, loss, ws)
            if row_major:
                faar.layer_step_rowmajor(ctx, faar.make_shape(O, K, T, ldxt=0, yref_transposed=1), hp, X, *state)
            else:
                faar.layer_step(ctx, shape, hp, X, Xt, *state)
        faar.check_status(ctx, ws)
        out.append((V, m, u, loss))
    assert all(torch.equal(a, b) for a, b in zip(*out)) and not torch.equal(out[0][0], V0)
