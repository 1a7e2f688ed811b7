"""Outputs whose rows are not whole 16-byte pieces (an odd N, an odd leading dimension, a base that is not 16-byte aligned):
the staged epilogue whose warps write the rows out.  Bit for bit on integer-valued inputs; GELU and SiLU through the gates
of tests/helpers.py; columns around the output stay untouched."""
import pytest
import torch

from tests.helpers import gates, oracle_for, small_int_inputs, to_f64
from paper_2604_26666_b200 import workloads as wl
from tests.test_gemm_gpu import ALL_EPI, h, mk  # noqa: F401

pytestmark = pytest.mark.gpu


def run_into(h, case, ins, ld, off, cfg=None):  # noqa: F811
    """The call with its output at element `off` of rows of `ld` elements; returns (result, everything around it intact)."""
    dt = torch.float32 if case.out == "f32" else torch.bfloat16
    flat = torch.full((case.M * ld + off + 64,), -7.0, dtype=dt, device="cuda")
    out = flat[off: off + case.M * ld].view(case.M, ld)[:, : case.N]
    dev = lambda t: None if t is None else t.cuda()
    h.linear(dev(ins.X), dev(ins.W), bias=dev(ins.bias), residual=dev(ins.residual), epilogue=case.epilogue, layout="NK",
             out=out, cfg=cfg)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    got = out.clone()
    out.fill_(-7.0)
    return got, bool((flat == -7.0).all())


# N odd, 1 past a chunk, below a chunk; even leading dimensions that are no multiple of 8, odd ones (every second row on a
# 2-byte boundary), bases off by one element; rows past M in the last tile, pairs and single CTAs
@pytest.mark.parametrize("epi", ALL_EPI)
@pytest.mark.parametrize("out", ["bf16", "f32"])
@pytest.mark.parametrize("N,ld,off", [(201, 201, 0), (257, 260, 0), (130, 130, 2), (128, 131, 1), (331, 333, 3), (64, 64, 1)])
def test_rows_of_any_alignment(h, epi, out, N, ld, off):  # noqa: F811
    case = mk(f"any_{epi}", 300, N, 520, epilogue=epi, layout="NK", out=out, w_scale=0.05)
    exact = epi not in ("BIAS_GELU_TANH", "SILU_GATE")
    ins = small_int_inputs(case, 12, lo=-2, hi=2) if exact else wl.make_inputs(case)
    ref = torch.from_numpy(oracle_for(ins, case))
    for cfg in (None, {"cta_group": 2, "tile_n": 256}, {"cta_group": 1, "tile_n": 64}):
        got, intact = run_into(h, case, ins, ld, off, cfg)
        assert intact
        if exact:
            assert torch.equal(got.cpu().double(), ref.to(got.dtype).double())
        else:
            c, t = gates(ref.numpy(), to_f64(got), out, epi)
            assert c <= 1 and t <= 1, (c, t)
        # the same bits as the register stores, which sum and round alike
        direct, _ = run_into(h, case, ins, ld, off, dict(cfg or {"cta_group": 2, "tile_n": 128}, store_mode=1))
        if exact:
            assert torch.equal(got, direct)


def test_batched_odd_strides_and_stream_k_choice(h):  # noqa: F811
    g = torch.Generator().manual_seed(4)
    A = torch.randint(-3, 4, (3, 140, 136), generator=g).to(torch.bfloat16)
    B = torch.randint(-3, 4, (3, 77, 136), generator=g).to(torch.bfloat16)
    ref = (A.double() @ B.double().transpose(1, 2)).to(torch.bfloat16)
    flat = torch.full((3, 140 * 79 + 5), -7.0, dtype=torch.bfloat16, device="cuda")
    out = flat[:, : 140 * 79].view(3, 140, 79)[:, :, :77]
    h.gemm_batched(A.cuda(), B.cuda(), layout="NK", out=out)
    assert torch.equal(out.cpu(), ref)
    out.fill_(-7.0)
    assert (flat == -7.0).all()
    # a stream-K choice runs data-parallel for an output that tensor stores cannot address
    X, W = torch.ones(300, 1024, dtype=torch.bfloat16).cuda(), torch.ones(601, 1024, dtype=torch.bfloat16).cuda()
    assert (h.gemm(X, W, layout="NK", cfg={"split_k": -1}) == 1024.0).all()
    # ... and asks for no scratch; an output of whole 16-byte pieces does
    assert h.workspace_bytes("gemm", 1, 300, 601, 1024, "NONE", "NK", cfg={"split_k": -1}) == 0
    assert h.workspace_bytes("gemm", 1, 300, 600, 1024, "NONE", "NK", cfg={"split_k": -1}) > 0
    assert h.device_status() == 0


@pytest.mark.parametrize("schedule", [1, 2])
def test_columns_beside_an_aligned_output_that_ends_inside_a_16_byte_piece(h, schedule):  # noqa: F811
    # rows 16-byte aligned and 16-byte multiples apart, N not: tensor stores would zero the columns behind the last one
    for out, N, ld in (("bf16", 257, 264), ("bf16", 260, 264), ("f32", 258, 260)):
        case = mk("ragged_piece", 700, N, 264, epilogue="BIAS", layout="NK", out=out)
        ins = small_int_inputs(case, 13, lo=-2, hi=2)
        ref = torch.from_numpy(oracle_for(ins, case))
        for cfg in ({"schedule": schedule, "cta_group": 1, "tile_n": 64}, {"schedule": schedule, "store_mode": 2},
                    {"split_k": -1}, {"split_k": 2}):
            if cfg.get("split_k") == 2:
                cfg = dict(cfg, cta_group=1)
            got, intact = run_into(h, case, ins, ld, 0, cfg)
            assert intact and torch.equal(got.cpu().double(), ref.to(got.dtype).double()), (out, cfg)


def test_row_sums_out_beside_a_ragged_last_piece(h):  # noqa: F811
    M, N, K = 200, 132, 128
    X, W = torch.ones(M, K, dtype=torch.bfloat16).cuda(), torch.ones(N, K, dtype=torch.bfloat16).cuda()
    wide = torch.full((M, 136), -7.0, dtype=torch.bfloat16, device="cuda")
    stats = torch.empty((N + 63) // 64, M, 2, device="cuda")
    h.linear(X, W, out=wide[:, :N], stats_out=stats)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    assert (wide[:, :N] == 128.0).all() and (wide[:, N:] == -7.0).all()
    assert (stats[:2, :, 0] == 64 * 128.0).all() and (stats[2, :, 0] == 4 * 128.0).all()
