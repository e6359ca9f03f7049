"""dK and dV of key tiles whose query tiles are dealt over the CTAs of a cluster (few key tiles) against the oracle: fewer items than
CTAs, rows and keys beyond the end, one head per key / value head, the values with which every CTA of a part finishes."""
import pytest

from paper_2603_22370_b200 import faar
from tests.test_gpu_attention import _attention_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2603_22370_b200 import build
    build.build()
    c = faar.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("B,S,H,HKV", [
    (1, 256, 1, 1),          # four items for the first key tile, two for the second: two parts
    (1, 449, 1, 1),          # eight: four parts, two of which have nothing of the last key tile's one item
    (2, 130, 4, 1),          # the last key tile holds two keys
    (1, 300, 8, 2),
    (1, 300, 16, 16),        # heads of 128: two parts, each finishing its columns in two turns, with the last key tile's rows cut inside a warp
])
def test_dealt_key_tiles_match_the_oracle(ctx, B, S, H, HKV, D):
    _attention_case(ctx, B, S, H, HKV, D)
