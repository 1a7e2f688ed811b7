"""GPU parity of attention where an item's second tile has no rows (sequences whose last 128-row tile is the first of its
item) and where sequences fit one tile and an item holds two heads, against the FP64 oracle under the gates of
test_attention_gpu."""
import numpy as np
import pytest

from tests.test_attention_gpu import check, h, rnd  # noqa: F401

pytestmark = pytest.mark.gpu


# more (batch, head) pairs than SMs: two heads per item (odd and even counts, grouped queries, several items per CTA); one,
# two and more key blocks; lengths at the edges of a block and of the tile
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("B,T,Hq,Hkv", [(151, 40, 1, 1), (25, 64, 6, 6), (19, 65, 8, 2), (40, 127, 12, 12), (13, 128, 12, 4),
                                        (170, 100, 2, 1), (300, 33, 3, 3)])
def test_two_heads_per_item(h, B, T, Hq, Hkv, D, causal):  # noqa: F811
    rows = np.array(sorted({0, 1, T // 2, T - 2, T - 1}), dtype=np.int64)
    check(h, rnd((B, T, Hq, D), 51), rnd((B, T, Hkv, D), 52), rnd((B, T, Hkv, D), 53), causal, rows=rows)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("Tq,Tk", [(100, 391), (128, 64), (77, 1)])
def test_two_heads_per_item_with_other_lengths_of_keys(h, Tq, Tk, D):  # noqa: F811
    check(h, rnd((38, Tq, 4, D), 54), rnd((38, Tk, 2, D), 55), rnd((38, Tk, 2, D), 56), False)


# a last item without a second tile: in every item (T <= 128, few heads), after and before items with both tiles, in several
# rounds (host's deal and closed form)
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("B,T,H", [(2, 100, 3), (3, 300, 2), (1, 384, 5), (16, 300, 12), (50, 260, 6), (5, 600, 12)])
def test_second_tile_without_rows(h, B, T, H, D, causal):  # noqa: F811
    rows = np.array(sorted({0, 1, 127, T // 2, T - 2, T - 1} & set(range(T))), dtype=np.int64)
    check(h, rnd((B, T, H, D), 57), rnd((B, T, H, D), 58), rnd((B, T, H, D), 59), causal, rows=rows)
