"""Launches that start, or ask for their operands, before the one before them has ended: what they read early has to be complete by then.
Every run is compared, bit for bit, with one in which each call waits for the one before it."""
import pytest
import torch

from paper_2603_22370_b200 import faar
from tests.test_gpu_model_passes import make_model

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


@pytest.mark.parametrize("O,K,T", [(64, 8192, 300), (128, 256, 1024), (512, 512, 512), (1000, 1040, 777), (512, 2048, 4096), (2048, 2048, 2048)])
@pytest.mark.parametrize("row_major", [False, True])
def test_a_step_takes_what_the_calls_before_it_wrote(ctx, O, K, T, row_major):
    """A step's products ask for X, X^T, the target and the optimiser state ahead.  Here the library's own calls (quantiser, transposition,
    frozen target, the step before) rewrite all of them directly before each step, from batches of very different values."""
    gen = torch.Generator(device=DEV).manual_seed(O + T)
    rnd = lambda r, c, s: (torch.randn((r, c), device=DEV, generator=gen) * s).to(torch.bfloat16)  # noqa: E731
    W, batches = rnd(O, K, 0.05), [rnd(T, K, s) for s in (0.3, 5.0, 1.0)]
    ldt = (T + 7) // 8 * 8
    shape = faar.make_shape(O, K, T, ldxt=ldt, yref_transposed=1)
    ws = torch.empty(faar.workspace_size(shape), dtype=torch.uint8, device=DEV)
    faar.workspace_init(ctx, ws)
    X, Xt = torch.empty((T, K), dtype=torch.bfloat16, device=DEV), torch.zeros((K, ldt), dtype=torch.bfloat16, device=DEV)
    Yref, sx = torch.zeros((O, shape.ldy), dtype=torch.bfloat16, device=DEV), torch.empty(1, device=DEV)
    scales, code = (torch.empty((O, n), dtype=torch.uint8, device=DEV) for n in (K // 16, K // 2))
    s_global, V0 = torch.empty(1, device=DEV), torch.empty((O, K), device=DEV)
    faar.softquant_init(ctx, shape, W, 0.0, scales, s_global, code, V0, ws)

    def run(wait):
        V, m, u, loss = V0.clone(), torch.zeros_like(V0), torch.zeros_like(V0), torch.zeros(2, device=DEV)
        losses = []
        torch.cuda.synchronize()
        for t in range(24):
            hp = faar.make_hparams(beta=5.0, lr=1e-2, step=t + 1, wsoft_ready=int(t % 4 == 3), beta_next=5.0 if t % 4 == 2 else 0.0)
            state = (Yref, V, code, scales, s_global, m, u, loss, ws)
            calls = [lambda: faar.layer_ref(ctx, shape, batches[t % 3], W, Yref, ws),
                     lambda: faar.act_fakequant(ctx, T, K, batches[t % 3], K, 0.0, X, K, sx, None, None, ws),
                     lambda: faar.transpose_bf16(ctx, T, K, X, K, Xt, ldt)]
            if row_major:
                calls = (calls[:2] if t % 2 else calls[1::-1]) + [lambda: faar.layer_step_rowmajor(ctx, shape, hp, X, *state)]
            else:
                calls = (calls if t % 2 else [calls[1], calls[2], calls[0]]) + [lambda: faar.layer_step(ctx, shape, hp, X, Xt, *state)]
            for call in calls:
                call()
                if wait:
                    torch.cuda.synchronize()
            losses.append(loss.clone())
        faar.check_status(ctx, ws)
        return [V, m, u] + losses

    want = run(True)
    for _ in range(5):
        assert all(torch.equal(a, b) for a, b in zip(run(False), want))


@pytest.mark.parametrize("batch,seq,hidden,heads,kv_heads,head_dim,ffn,layers", [
    (2, 96, 128, 2, 1, 64, 256, 3), (1, 300, 512, 8, 2, 64, 1024, 2), (2, 500, 512, 4, 2, 128, 1040, 2), (1, 129, 2048, 16, 4, 128, 2048, 1)])
def test_a_models_steps_with_launches_next_to_one_another(ctx, batch, seq, hidden, heads, kv_heads, head_dim, ffn, layers):
    """The same steps with an event behind every launch, which nothing starts ahead of: dW products next to input gradients and dQ next to
    dK / dV read and write nothing of one another."""
    runs = []
    for apart in (True, False, False, False):
        m, tokens, _ = make_model(ctx, batch, seq, vocab=528, hidden=hidden, n_layers=layers, n_heads=heads, n_kv_heads=kv_heads, head_dim=head_dim,
                                  ffn=ffn)
        losses = []
        torch.cuda.synchronize()
        if apart:
            faar.profile_begin(ctx)
        for t in range(6):
            m.step(tokens, beta=4.0 + t, lr=1e-2)
            losses.append(m.loss.clone())
        if apart:
            faar.profile_end(ctx)
        faar.check_status(ctx, m.ws)
        runs.append(losses + [x.V for lins in m.lin for x in lins.values()])
    for other in runs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(runs[0], other))
