"""Products of fewer rows than a tile load only those rows: every kernel that shares the load, at the edges of the box (multiples
of 8 rows, one row, one less than a tile), exact on integers, whatever an earlier product left in shared memory."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    from paper_2604_26666_b200.binding import Handle
    hd = Handle(0)
    yield hd
    hd.close()


def ints(shape, seed, dtype=torch.bfloat16):
    g = torch.Generator().manual_seed(seed)
    return torch.randint(-3, 4, shape, generator=g).float().to(dtype).cuda()


def dirty(h):
    """Leaves infinities and NaNs in the operand stages."""
    bad = torch.full((2048, 512), float("inf"), dtype=torch.bfloat16, device="cuda")
    h.gemm(bad, bad, layout="NK")


@pytest.mark.parametrize("M", [1, 7, 8, 9, 20, 64, 113, 120, 121, 127, 128])
def test_few_rows(h, M):
    K, N = 656, 264
    X, W = ints((M, K), M), ints((N, K), 1)
    ref = X.float() @ W.float().t()
    for cfg in (None, dict(cta_group=1, tile_n=64), dict(cta_group=1, tile_n=256), dict(cta_group=2, tile_n=128), dict(cta_group=1, tile_n=64, split_k=3),
                dict(cta_group=1, tile_n=64, split_k=2, schedule=3), dict(cta_group=1, tile_n=64, split_k=-1)):
        dirty(h)
        assert torch.equal(h.gemm(X, W, layout="NK", out_dtype=torch.float32, cfg=cfg), ref), cfg
    dirty(h)
    assert torch.equal(h.gemm_splitk(X, W, layout="NK"), ref)
    Xb, Wb = ints((3, M, K), M + 1), ints((3, N, K), 2)
    dirty(h)
    assert torch.equal(h.gemm_batched(Xb, Wb, layout="NK", out_dtype=torch.float32), Xb.float() @ Wb.float().transpose(1, 2))
    X8, W8 = ints((M, K), M + 2, torch.float8_e4m3fn), ints((N, K), 3, torch.float8_e4m3fn)
    dirty(h)
    assert torch.equal(h.linear_fp8(X8, W8, 1.0, out_dtype=torch.float32), X8.float() @ W8.float().t())
    assert h.device_status() == 0
