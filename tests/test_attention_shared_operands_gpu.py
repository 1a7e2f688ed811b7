"""Attention whose batch entries share one query, key or value tensor (batch stride 0, as expand() makes it): the same bits
as with a copy per entry, on every path of the dispatch; an output that all entries would share is refused."""
import pytest
import torch

from tests.test_attention_gpu import h, rnd  # noqa: F401  (h is the fixture)

pytestmark = pytest.mark.gpu


# few query rows (one CTA a head, and clusters); head_dim 64: two tiles an SM, three, pairs of heads, pairs of tiles, dealt
# tiles; head_dim 128: halves, pairs of heads, pairs of tiles in closed form and dealt
@pytest.mark.parametrize("B,Tq,Tk,Hq,Hkv,D,causal", [
    (3, 1, 200, 8, 2, 128, False), (2, 4, 900, 4, 4, 64, False),
    (2, 100, 100, 4, 2, 64, True), (16, 64, 64, 12, 12, 64, False), (16, 128, 128, 12, 12, 64, True),
    (40, 300, 200, 12, 4, 64, False), (16, 500, 500, 12, 12, 64, True),
    (2, 100, 70, 8, 2, 128, False), (8, 100, 100, 32, 8, 128, True), (2, 300, 300, 4, 2, 128, False), (5, 512, 512, 32, 8, 128, True)])
def test_shared_operands_are_copies_of_one(h, B, Tq, Tk, Hq, Hkv, D, causal):  # noqa: F811
    q, k, v = rnd((B, Tq, Hq, D), 41).cuda(), rnd((B, Tk, Hkv, D), 42).cuda(), rnd((B, Tk, Hkv, D), 43).cuda()
    one = lambda t: t[:1].expand(t.shape)  # noqa: E731
    for a in ((q, one(k), one(v)), (one(q), k, v), (q, k, one(v))):
        assert torch.equal(h.attention(*a, causal=causal), h.attention(*(t.contiguous() for t in a), causal=causal))
    assert h.device_status() == 0


def test_a_shared_output_is_refused(h):  # noqa: F811
    from paper_2604_26666_b200.binding import FactError

    for Tq in (1, 200):
        q, out = rnd((2, Tq, 2, 64), 44).cuda(), torch.empty(1, Tq, 2, 64, dtype=torch.bfloat16, device="cuda")
        n = h.launch_count()
        with pytest.raises(FactError):
            h.attention(q, q, q, causal=False, out=out.expand(2, Tq, 2, 64))
        assert h.launch_count() == n
        h.attention(q[:1], q[:1], q[:1], causal=False, out=out)
