"""Calls with fewer routed items than SMs, whose weight tiles are cut to half of the full height: widths
around the multiples of 64, 128 and 256 rows, on single CTAs, CTA pairs and with a k-split reduction.
(The heights themselves: test_ffn_walk.py.)"""
import pytest

from paper_2505_19645_b200 import workloads as wl
from parity_utils import check_layer_against_oracle

pytestmark = pytest.mark.gpu


IDLE_TILE_CASES = [
    (256, 8, 2, 512, 0, 5),
    (288, 2, 1, 96, 0, 6),       # a 32-row rest in both passes
    (224, 3, 2, 160, 96, 33),
    (544, 4, 2, 64, 0, 128),
    (256, 1, 1, 2176, 0, 40),    # chunks of the reduction times few tiles
    (288, 2, 2, 160, 64, 129),   # pairs: tiles of twice the height
    (96, 4, 2, 352, 0, 260),
    (544, 20, 2, 160, 0, 40),    # low down tiles and full gate/up tiles
    (800, 16, 2, 96, 0, 130),    # low gate/up tiles, down tiles of full height on pairs: 512 and 288
]


@pytest.mark.parametrize("H,E,k,I,Is,T", IDLE_TILE_CASES)
def test_few_items_match_the_oracle(H, E, k, I, Is, T):
    shape = wl.small_shape("idle", H, E, k, I, Is, 0, 1, 1 if Is else 0)
    w = wl.make_weights(shape, 300 + H + T, "cuda")
    x = wl.make_tokens(shape, T, 400 + T, "cuda")
    check_layer_against_oracle(shape, w, x, T, 0)
