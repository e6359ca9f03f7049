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
])
def test_dealt_key_tiles_match_the_oracle(ctx, B, S, H, HKV, D):
    _attention_case(ctx, B, S, H, HKV, D)


def test_two_parts_whose_columns_take_two_turns(ctx):
    """Heads of 128 and as many key tiles as leave room for two parts: each finishes its columns in two turns, here with the last key
    tile's rows ending inside a warp."""
    _attention_case(ctx, 1, 300, 16, 16, 128)
