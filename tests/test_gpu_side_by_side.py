"""Launches that run next to the one before them: dQ next to dK / dV, unless dq lies over something that kernel still reads."""
import pytest
import torch

from paper_2603_22370_b200 import faar

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("over", ["q", "dout"])
@pytest.mark.parametrize("B,S,H,HKV,D", [(2, 300, 4, 2, 64), (1, 700, 2, 1, 128)])
def test_dq_may_take_the_place_of_an_input(B, S, H, HKV, D, over):
    ctx = faar.Context(0)
    gen = torch.Generator(device=DEV).manual_seed(S)
    T, ld, ldk = B * S, H * D, HKV * D
    rnd = lambda *s: torch.randn(s, device=DEV, generator=gen).to(torch.bfloat16)  # noqa: E731
    q, k, v, dout = rnd(T, ld), rnd(T, ldk), rnd(T, ldk), rnd(T, ld)
    out, lse, dsum = torch.empty_like(q), torch.empty(T * H, device=DEV), torch.empty(T * H, device=DEV)
    faar.attention_fwd(ctx, B, S, H, HKV, D, q, ld, k, v, ldk, out, ld, lse)
    want = [torch.empty_like(t) for t in (q, k, v)]
    faar.attention_bwd(ctx, B, S, H, HKV, D, q, ld, k, v, ldk, out, dout, ld, lse, dsum, *want)
    for _ in range(20):
        args = {"q": q.clone(), "dout": dout.clone()}
        got = [args[over], torch.empty_like(k), torch.empty_like(v)]
        faar.attention_bwd(ctx, B, S, H, HKV, D, args["q"], ld, k, v, ldk, out, args["dout"], ld, lse, dsum, *got)
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    faar.attention_status(ctx)
    ctx.close()
