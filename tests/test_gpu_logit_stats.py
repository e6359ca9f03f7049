"""The alignment loss from the softmax statistics that the logits' products leave behind, against the loss that reads the logits for
them: a last tile of 16 columns, one row more than a row block, whole tiles; a temperature other than 1."""
import pytest
import torch

from paper_2603_22370_b200 import faar
from tests.test_gpu_model_passes import ctx, make_model  # noqa: F401

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("tau", [1.0, 1.7])
@pytest.mark.parametrize("batch,seq,vocab", [(1, 257, 18944), (2, 150, 9488), (4, 256, 8192), (1, 129, 18960)])
def test_loss_from_the_products_statistics(ctx, batch, seq, vocab, tau):  # noqa: F811
    m, tokens, _ = make_model(ctx, batch, seq, vocab=vocab, hidden=64, n_layers=1, n_heads=1, n_kv_heads=1, head_dim=64, ffn=64)
    T, d = batch * seq, 64
    n = faar.logit_stats_size(ctx, T, vocab)
    assert n == T * ((vocab + 127) // 128) * 8
    Z_fp, H_fp, _ = m.forward(tokens, quantised=False)
    Z, H, _ = m.forward(tokens, quantised=True, beta=6.0)
    stats = [torch.full((n,), 0xFF, dtype=torch.uint8, device=DEV) for _ in range(2)]
    again = m._forward(m._table(), tokens, False, tau=tau, stats=stats[0])[:2] + m._forward(m._table(), tokens, True, 6.0, tau=tau, stats=stats[1])[:2]
    assert all(torch.equal(a, b) for a, b in zip(again, (Z_fp, H_fp, Z, H)))
    out = []
    for given in (False, True):
        dZ, dH, loss = torch.empty_like(Z), torch.empty_like(H), torch.zeros(2, device=DEV)
        args = (ctx, T, vocab, d, Z_fp, Z, vocab, H_fp, H, d, tau, 0.9)
        if given:
            faar.align_loss_stats(*args, *stats, dZ, dH, loss, m.aws)
        else:
            faar.align_loss(*args, dZ, dH, loss, m.aws)
        out.append((dZ.double(), dH, loss.double()))
    faar.check_status(ctx, m.ws)
    (dZ0, dH0, l0), (dZ1, dH1, l1) = out
    assert torch.equal(dH0, dH1) and l0[1] == l1[1]
    # a row's log-sum-exp, an FP32 number of up to 32 (a unit of 2^-19), from sums in another order: a few units, which is as much of
    # each probability; the gradient is the difference of two and may round to the next BF16 (2^-7 of it)
    P = torch.softmax(Z.double() / tau, -1) + torch.softmax(Z_fp.double() / tau, -1)
    assert torch.all((dZ0 - dZ1).abs() <= 2.0**-7 * dZ0.abs() + 2.0**-17 * (0.9 / (tau * T)) * P)
    # the loss: a sum of P_fp (log P_fp - log P_q), whose terms move by the units of both
    assert abs(l0[0] - l1[0]) <= 2.0**-16 * max(1.0, float(l0[0]))


def test_small_products_leave_none(ctx):  # noqa: F811
    assert faar.logit_stats_size(ctx, 192, 512) == 0 and faar.logit_stats_size(ctx, 128, 128256) == 0
    m, tokens, _ = make_model(ctx, 1, 32, vocab=528, hidden=64, n_layers=1, n_heads=1, n_kv_heads=1, head_dim=64, ffn=64)
    stats = torch.zeros(1 << 16, dtype=torch.uint8, device=DEV)
    with pytest.raises(faar.FaarError) as e:
        m._forward(m._table(), tokens, False, stats=stats)
    assert e.value.status == faar.ERR_SHAPE
    with pytest.raises(faar.FaarError) as e:
        m._forward(m._table(), tokens, False, tau=0.0, stats=stats)
    assert e.value.status == faar.ERR_INVALID_ARG


def test_buffers_and_products_that_the_statistics_calls_refuse(ctx):  # noqa: F811
    """A buffer for fewer tokens or a smaller vocabulary, in any of the calls, and a loss on statistics that no product leaves.  Every
    refusal comes from a comparison on the host: nothing is launched."""
    batch, seq, vocab, d = 1, 257, 18944, 64
    m, tokens, _ = make_model(ctx, batch, seq, vocab=vocab, hidden=d, n_layers=1, n_heads=1, n_kv_heads=1, head_dim=64, ffn=64)
    n = faar.logit_stats_size(ctx, seq, vocab)
    Z, H = (torch.zeros((seq, c), dtype=torch.bfloat16, device=DEV) for c in (vocab, d))
    arena = {k: torch.empty(m.arena_bytes[k], dtype=torch.uint8, device=DEV) for k in (False, True)}
    whole, short = (torch.zeros(k, dtype=torch.uint8, device=DEV) for k in (n, n - 1))
    table, loss = m._table(), torch.zeros(2, device=DEV)

    def forward(s):
        faar.model_forward_stats(ctx, table, batch, seq, tokens, m.pos, False, 4.0, False, arena[False], Z, H, 1.0, s, m.ws)

    def both(s_fp, s):
        faar.model_forward_both_stats(ctx, table, batch, seq, tokens, m.pos, 4.0, arena[False], Z, H, arena[True], Z, H, 1.0, s_fp, s, m.ws)

    def align(s_fp, s, T=seq, V=vocab):
        faar.align_loss_stats(ctx, T, V, d, Z, Z, vocab, H, H, d, 1.0, 1.0, s_fp, s, None, None, loss, m.aws)

    for call, status in [(lambda: forward(short), faar.ERR_WORKSPACE), (lambda: both(whole, short), faar.ERR_WORKSPACE),
                         (lambda: both(short, whole), faar.ERR_WORKSPACE), (lambda: align(whole, short), faar.ERR_WORKSPACE),
                         (lambda: align(short, whole), faar.ERR_WORKSPACE), (lambda: align(whole, None), faar.ERR_INVALID_ARG),
                         (lambda: forward(None), faar.ERR_INVALID_ARG), (lambda: align(whole, whole, T=128), faar.ERR_SHAPE),
                         (lambda: align(whole, whole, V=vocab - 8), faar.ERR_SHAPE), (lambda: align(whole[8:], whole), faar.ERR_ALIGN)]:
        with pytest.raises(faar.FaarError) as e:
            call()
        assert e.value.status == status
    align(whole, whole)
    torch.cuda.synchronize()
    faar.check_status(ctx, m.ws)


@pytest.mark.parametrize("T,vocab,fit,pay", [
    (511, 128256, True, False),           # few tokens, whatever the vocabulary
    (512, 12544, True, False),            # 98 tiles of 256 x 256
    (512, 12800, True, True),             # 100
    (999, 6144, True, False),
    (1000, 4736, True, True),             # 76
    (1000, 4608, False, False),           # 72: not a tile for every CTA pair
    (4096, 1192, False, False),           # not a multiple of 16
])
def test_where_statistics_pay(ctx, T, vocab, fit, pay):  # noqa: F811
    assert (faar.logit_stats_size(ctx, T, vocab) > 0, faar.logit_stats_pay(ctx, T, vocab)) == (fit, pay)


@pytest.mark.parametrize("tau", [1.0, 1.7])
@pytest.mark.parametrize("T,vocab", [(513, 8720), (1000, 4736)])      # a last slot of 16 columns; whole slots
def test_a_step_is_the_same_whatever_is_handed_in_or_out(ctx, T, vocab, tau):  # noqa: F811
    """Losses and every V of a plain step, passes next to one another or in turn, of one that returns its gradients, and of one on frozen
    outputs formed before: statistics or not is one choice for all."""
    assert faar.logit_stats_pay(ctx, T, vocab)
    runs = []
    for overlap, want_dv, given in [(True, False, False), (False, False, False), (True, True, False), (False, True, False), (True, False, True),
                                    (False, True, True)]:
        m, tokens, _ = make_model(ctx, 1, T, vocab=vocab, hidden=64, n_layers=1, n_heads=1, n_kv_heads=1, head_dim=64, ffn=64)
        m.overlap = overlap
        fp = m.forward(tokens, quantised=False)[:2] if given else None
        m.step(tokens, beta=6.0, tau=tau, lambda_kl=0.9, want_dv=want_dv, fp_outputs=fp)
        faar.check_status(ctx, m.ws)
        runs.append([m.loss.clone()] + [x.V for lins in m.lin for x in lins.values()])
    for other in runs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(runs[0], other))


@pytest.mark.parametrize("T,vocab,ldz", [(257, 18960, 18960), (300, 9472, 9480)])
def test_statistics_of_logits_that_are_there(ctx, T, vocab, ldz):  # noqa: F811
    """Maximum and sum of every 128 columns against 64 bits, with a minute and an infinite logit and a row that is all alike."""
    gen = torch.Generator(device=DEV).manual_seed(T)
    Z = torch.full((T, ldz), float("nan"), dtype=torch.bfloat16, device=DEV)
    Z[:, :vocab] = (torch.randn((T, vocab), device=DEV, generator=gen) * 4).to(torch.bfloat16)
    Z[0, 5], Z[1, 130], Z[2, :vocab] = -3.0e38, float("-inf"), 1.5
    stats = torch.full((faar.logit_stats_size(ctx, T, vocab),), 0xFF, dtype=torch.uint8, device=DEV)
    faar.logit_stats(ctx, T, vocab, Z, ldz, 1.7, stats)
    got = stats.view(torch.float32).view(T, -1, 2).double()
    y = torch.full((T, got.shape[1] * 128), float("-inf"), dtype=torch.float64, device=DEV)
    y[:, :vocab] = Z[:, :vocab].double() * (1.4426950408889634 / 1.7)
    y = y.view(T, -1, 128)
    m = y.max(-1).values
    # the maximum is one rounding of the product with a rounded constant (2^-23 of it); the sum has that error in each of its exponents, the
    # hardware exponential's (2^-22) and up to 128 additions (2^-17)
    assert torch.all((got[..., 0] - m).abs() <= 2.0**-23 * m.abs())
    s = torch.exp2(y - got[..., :1]).sum(-1)
    assert torch.all((got[..., 1] - s).abs() <= (2.0**-17 + 2.0**-21 + 2.0**-22 * y[y.isfinite()].abs().clamp(max=2.0**7).max()) * s)
