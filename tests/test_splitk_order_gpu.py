"""The order of a split-K reduction, bit for bit: L >= 4 sums over slices q, q + L, ..., combined pairwise (so that no chain
is longer than a quarter of the slices).  Every slice's partial sum is one BF16 value, exact in FP32, and the values'
exponents are spread over 24 binades, so that another order shows."""
import numpy as np
import pytest
import torch

from tests.test_gemm_gpu import h  # noqa: F401

pytestmark = pytest.mark.gpu


def sums(parts, L):
    """parts [slices, ...] FP32 added up by L lanes."""
    lanes = [np.zeros(parts.shape[1:], np.float32) for _ in range(L)]
    for s, p in enumerate(parts):
        lanes[s % L] = lanes[s % L] + p
    while len(lanes) > 1:
        lanes = [a + b for a, b in zip(lanes[::2], lanes[1::2])]
    return lanes[0]


@pytest.mark.parametrize("M,N,K", [(256, 256, 131072), (256, 256, 524288), (80, 128, 209992), (200, 256, 83512), (64, 64, 16384)])
def test_four_or_more_lanes_add_the_slices_up(h, M, N, K):  # noqa: F811
    S = h.get_config("gemm_splitk", 1, M, N, K, out_dtype=torch.float32).split_k
    assert S > 8
    blocks = -(-K // 64)
    first = [64 * (s * (blocks // S) + min(s, blocks % S)) for s in range(S)]
    g = torch.Generator().manual_seed(S)
    part = (torch.randn(S, N, generator=g) * torch.exp2(torch.randint(-12, 13, (S, N), generator=g))).to(torch.bfloat16)
    A, B = torch.zeros(M, K, dtype=torch.bfloat16), torch.zeros(K, N, dtype=torch.bfloat16)
    A[:, first] = 1.0
    B[first] = part
    got = h.gemm_splitk(A.cuda(), B.cuda()).cpu().numpy()
    assert any((got == sums(part.float().numpy(), L)).all() for L in (4, 8, 16, 32))
    assert not (got == sums(part.float().numpy(), 1)).all()  # (the inputs tell orders apart)
    assert h.device_status() == 0
