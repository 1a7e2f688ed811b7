"""GPU parity of attention with few query rows per key/value head (decode) against the FP64 attention oracle, under the
gates of the other attention tests (derived in test_attention_gpu.attention_gates: probabilities and result rounded to
BF16; this path rounds in the same places)."""
import pytest
import torch

from tests.test_attention_gpu import attention_gates, check, h, rnd  # noqa: F401  (h is the fixture)
from tests.helpers import to_f64

pytestmark = pytest.mark.gpu


# one key, a warp's 16 keys and a 64-key block less, exactly and more, several blocks; one to eight CTAs per head
# (many or few (batch, head) pairs); rows below, at and above each group of 8 up to the limit of 32 and one past it
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("B,Tq,Tk,Hq,Hkv", [
    (1, 1, 1, 1, 1), (2, 1, 15, 3, 3), (1, 1, 17, 8, 2), (1, 1, 63, 4, 1), (1, 1, 64, 9, 1), (1, 1, 65, 8, 1),
    (1, 3, 129, 4, 2), (2, 8, 200, 4, 4), (1, 1, 1000, 32, 8), (3, 4, 515, 16, 4), (1, 17, 391, 2, 2),
    (1, 8, 700, 8, 2), (1, 32, 333, 2, 2), (1, 33, 333, 2, 2), (160, 1, 77, 2, 1), (20, 1, 260, 16, 4),
    (1, 32, 833, 8, 8), (4, 1, 705, 24, 12), (12, 2, 770, 4, 4)])
def test_few_query_rows(h, B, Tq, Tk, Hq, Hkv, D):  # noqa: F811
    check(h, rnd((B, Tq, Hq, D), 31), rnd((B, Tk, Hkv, D), 32), rnd((B, Tk, Hkv, D), 33), False)


@pytest.mark.parametrize("D", [64, 128])
def test_views_large_scores_and_repeatability(h, D):  # noqa: F811
    # keys and values inside one interleaved cache, the output inside a wider tensor; scores of size 36 (the reference
    # maximum moves often); repeated calls give the same bits
    B, Tq, Tk, Hq, Hkv = 2, 2, 450, 4, 2
    q, kv = rnd((B, Tq, Hq, D), 34, 6.0), rnd((B, Tk, 2 * Hkv, D), 35, 6.0)
    k, v = kv[:, :, :Hkv], kv[:, :, Hkv:]
    kvd = kv.cuda()
    wide = torch.full((B, Tq, Hq + 1, D), -7.0, dtype=torch.bfloat16, device="cuda")
    outs = []
    for _ in range(3):
        h.attention(q.cuda(), kvd[:, :, :Hkv], kvd[:, :, Hkv:], causal=False, out=wide[:, :, :Hq])
        torch.cuda.synchronize()
        outs.append(wide.clone())
    assert h.device_status() == 0
    assert all(torch.equal(outs[0], o) for o in outs[1:])
    assert (wide[:, :, Hq] == -7.0).all()
    c, t = attention_gates(q, k, v, False, to_f64(wide[:, :, :Hq]))
    # (values of size 6: the contract's absolute 1e-2 is meant for unit variance, the tight gate is the derived one)
    assert t <= 1.0, (c, t)


# many problems of few keys go to the tile kernels: a query row's bits are then those of a call with more rows than the
# few-rows kernel takes (every head size's kernels: two and three tiles an SM, halves, pairs of heads)
@pytest.mark.parametrize("B,Tq,Tk,Hq,Hkv,D", [(40, 32, 40, 12, 12, 64), (64, 17, 256, 12, 12, 64), (300, 1, 64, 12, 12, 64),
                                              (256, 8, 33, 8, 2, 64), (40, 32, 16, 12, 12, 128), (64, 20, 130, 8, 8, 128),
                                              (64, 8, 64, 32, 8, 128), (3, 32, 200, 32, 32, 128)])
def test_many_problems_of_few_keys_go_to_the_tiles(h, B, Tq, Tk, Hq, Hkv, D):  # noqa: F811
    q, k, v = rnd((B, 33, Hq, D), 36), rnd((B, Tk, Hkv, D), 37), rnd((B, Tk, Hkv, D), 38)
    few = h.attention(q[:, :Tq].contiguous().cuda(), k.cuda(), v.cuda(), causal=False)
    more = h.attention(q.cuda(), k.cuda(), v.cuda(), causal=False)
    assert h.device_status() == 0 and torch.equal(few, more[:, :Tq])
    c, t = attention_gates(q[:4, :Tq], k[:4], v[:4], False, to_f64(few[:4]))
    assert c <= 1.0 and t <= 1.0, (c, t)
