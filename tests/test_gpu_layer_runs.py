"""Runs of a layer on the batch as it is (short ones) and on its transposed copy (long ones): the same bits."""
import pytest
import torch

from paper_2603_22370_b200 import faar, inputs, stage1
from tests.gpu_helpers import dev_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("quantise_activations", [False, True])
@pytest.mark.parametrize("O,K,T,opt", [(64, 128, 96, 1), (130, 144, 603, 1), (300, 1040, 777, 0), (512, 2048, 1100, 1)])
def test_both_ways_through_a_layer_give_the_same_bits(monkeypatch, O, K, T, opt, quantise_activations):
    """The driver's own transposed copy, with padded rows where the tokens are no multiple of 8 or 16, of X or of its quantised values."""
    ctx = faar.Context(0)
    W, X = (dev_bf16(a) for a in inputs.config2(O, O, K, T))
    out = []
    for limit in (stage1.ROW_MAJOR_STEPS, 0):
        monkeypatch.setattr(stage1, "ROW_MAJOR_STEPS", limit)
        out.append(stage1.optimise_layer(ctx, W, X, steps=7, opt=opt, lr=1e-2 if opt else 1e-4, loss_every=2, quantise_activations=quantise_activations))
    a, b = out
    assert all(torch.equal(a[k], b[k]) for k in ("packed", "scales", "V", "s_global"))
    assert a["history"] == b["history"] and len(a["history"]) == 4
    ctx.close()
