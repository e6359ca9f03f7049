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
