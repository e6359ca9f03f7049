"""A model's passes in the bounds-checking build of the library (libfaar_debug.so): the epilogues that are theirs alone (the gated
product and its backward, rotary embedding, the logits' softmax statistics, the row sums of the attention's gradient in two, four and
eight parts, of a split contraction too) report no store outside its tensor and give the bits of the normal build."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import sys, numpy as np, torch
sys.path.insert(0, sys.argv[1])
from paper_2603_22370_b200 import faar, stage2
from tests.test_gpu_model_passes import make_model
ctx = faar.Context(0)
out = {}
for i, (batch, seq, vocab, hidden, heads, kv, dim, ffn) in enumerate([
        (1, 1000, 4752, 64, 1, 1, 64, 16), (2, 65, 528, 128, 2, 1, 64, 80), (3, 100, 528, 1024, 3, 3, 128, 336), (2, 500, 528, 512, 4, 2, 128, 1040),
        (1, 7, 64, 64, 1, 1, 64, 16)]):
    m, tokens, _ = make_model(ctx, batch, seq, vocab=vocab, hidden=hidden, n_layers=1, n_heads=heads, n_kv_heads=kv, head_dim=dim, ffn=ffn)
    assert faar.logit_stats_pay(ctx, batch * seq, vocab) == (i == 0)
    res = m.step(tokens, beta=6.0, want_dv=True)
    faar.check_status(ctx, m.ws)                       # raises if a checked store was out of range
    out[str(i)] = np.concatenate([m.loss.cpu().numpy(), res["Z_q"].float().cpu().numpy().ravel()] + [g.cpu().numpy().ravel() for g in res["dV"].values()])
np.savez(sys.argv[2], **out)
print("child ok", faar.LIB_PATH)
'''


def test_a_models_passes_in_the_bounds_checking_build(tmp_path):
    from paper_2603_22370_b200 import build
    got = {}
    for lib in (build.build(debug=True), build.build()):
        path = str(tmp_path / (os.path.basename(lib) + ".npz"))
        res = subprocess.run([sys.executable, "-c", CHILD, ROOT, path], env=dict(os.environ, FAAR_LIB=lib), capture_output=True, text=True, timeout=600)
        assert res.returncode == 0 and lib in res.stdout, res.stdout[-2000:] + res.stderr[-4000:]
        got[lib] = np.load(path)
    dbg, ref = got.values()
    assert sorted(dbg.files) == sorted(ref.files) and len(ref.files) == 5
    assert all(np.array_equal(dbg[k], ref[k]) for k in ref.files)
