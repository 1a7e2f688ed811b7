"""Linear layers of few rows (at most 64): the kernel that streams the weights (schedule 4), against the oracle.  Bit for
bit on integer-valued inputs where the epilogue is exact on integers, through the gates of the other GEMM tests
(tests/helpers.py) for GELU and SiLU."""
import pytest
import torch

from paper_2604_26666_b200 import workloads as wl
from tests.test_gemm_gpu import bit_exact, check_case, h, mk, oracle_for, run_gpu, small_int_inputs  # noqa: F401

pytestmark = pytest.mark.gpu


# rows at the edges of the groups of 8 and of the 8 / 16 / 32 / 64 variants; N below, at and past a CTA's weight rows, odd
# (stored element by element); K below one box of 64, ragged in the last box and in the last stage, several ring turns
@pytest.mark.parametrize("tile_n", [16, 32, 64])
@pytest.mark.parametrize("layout", ["NK", "KN"])
@pytest.mark.parametrize("M,N,K", [(1, 32, 8), (7, 72, 64), (8, 48, 200), (9, 200, 264), (16, 336, 1000), (17, 40, 520),
                                   (32, 72, 768), (33, 136, 264), (64, 520, 4104), (5, 8, 16384)])
def test_every_variant_is_exact_on_integers(h, tile_n, layout, M, N, K):  # noqa: F811
    if layout == "KN" and tile_n == 16:
        pytest.skip("rows of 32 bytes are not loaded from a [K, N] operand")
    for epi, out in (("NONE", "f32"), ("BIAS_RESIDUAL", "bf16"), ("BIAS_RELU", "f32")):
        case = mk(f"few_{epi}", M, N, K, epilogue=epi, layout=layout, out=out)
        bit_exact(h, case, small_int_inputs(case, 5, lo=-2, hi=2), cfg={"schedule": 4, "tile_n": tile_n})


@pytest.mark.parametrize("M", [1, 12, 30, 64])
@pytest.mark.parametrize("epi", ["BIAS_GELU_TANH", "SILU_GATE", "BIAS"])
def test_the_library_chooses_it_and_the_epilogues_hold(h, M, epi):  # noqa: F811
    for N, K in ((200, 776), (2400, 256)):  # (16 and 32 weight rows per CTA; half of them gate rows)
        case = mk(f"few_{epi}", M, N, K, epilogue=epi, layout="NK", w_scale=0.05)
        assert h.get_config("linear", 1, M, N, K, epi, "NK").schedule == 4
        assert h.workspace_bytes("linear", 1, M, N, K, epi, "NK") == 0
        check_case(h, case)
    assert h.get_config("linear", 1, 65, 200, 776, epi, "NK").schedule != 4


def test_odd_widths_strided_outputs_and_repeatability(h):  # noqa: F811
    M, N, K = 6, 101, 1032
    case = mk("few_odd", M, N, K, op="gemm", layout="NK")
    ins = small_int_inputs(case, 8, lo=-2, hi=2)
    ref = torch.from_numpy(oracle_for(ins, case)).to(torch.bfloat16)
    wide = torch.full((M, N + 3), -7.0, dtype=torch.bfloat16, device="cuda")
    for _ in range(3):
        h.gemm(ins.X.cuda(), ins.W.cuda(), layout="NK", out=wide[:, :N])
        torch.cuda.synchronize()
        assert torch.equal(wide[:, :N].cpu(), ref) and (wide[:, N:] == -7.0).all()
    real = wl.make_inputs(mk("few_real", 16, 768, 3072, layout="NK", w_scale=0.05))
    c2 = mk("few_real", 16, 768, 3072, layout="NK", w_scale=0.05)
    first = run_gpu(h, real, c2).clone()
    assert all(torch.equal(first, run_gpu(h, real, c2)) for _ in range(3))
    assert h.device_status() == 0


def test_what_it_does_not_serve_is_refused_or_goes_elsewhere(h):  # noqa: F811
    from paper_2604_26666_b200.binding import FactError

    X, W = torch.ones(8, 128, dtype=torch.bfloat16).cuda(), torch.ones(256, 128, dtype=torch.bfloat16).cuda()
    for bad in ({"schedule": 4, "split_k": 2}, {"schedule": 4, "tile_n": 48}, {"schedule": 4, "stages": 40},
                {"schedule": 4, "store_mode": 2}):
        with pytest.raises(FactError):
            h.linear(X, W, cfg=bad)
    with pytest.raises(FactError):
        h.linear(X.repeat(9, 1), W, cfg={"schedule": 4})
    stats = torch.empty(4, 8, 2, device="cuda")
    y = h.linear(X, W, stats_out=stats)  # (row sums out: the tile kernel)
    assert (y == 128.0).all() and (stats[..., 0] == 64 * 128.0).all()
    assert (h.linear(X, W.t().contiguous(), layout="KN", epilogue="SILU_GATE") > 0).all()


def test_a_tuned_entry_is_for_plain_calls_only(h, tmp_path):  # noqa: F811
    # the table's key is the shape: calls of it that the kernel does not serve take the library's own choice
    from paper_2604_26666_b200.binding import Handle

    M, N, K = 8, 256, 128
    X, W = torch.ones(M, K, dtype=torch.bfloat16).cuda(), torch.ones(N, K, dtype=torch.bfloat16).cuda()
    path = tmp_path / "table.txt"
    for entry in ("8 16 64 4 1 1 1 1 4", "128 64 64 4 1 1 2 0 3"):  # few rows; K slices as a cluster
        path.write_text(f"3 0 1 0 1 {M} {N} {K} | {entry}\n")
        t = Handle(0, load_table=False)
        t.tune_cache_load(str(path))
        assert t.get_config("linear", 1, M, N, K, "NONE", "NK").schedule == int(entry[-1])
        assert (t.linear(X, W) == K).all()
        stats = torch.empty(N // 64, M, 2, device="cuda")
        assert (t.linear(X, W, stats_out=stats) == K).all() and (stats[..., 0] == 64 * K).all()
        folded = t.linear(X, W, x_norm="rms", x_stats=t.row_stats(X), eps=0.0)
        assert torch.allclose(folded.float(), torch.full_like(folded, K).float(), rtol=2 ** -7)
        assert (t.linear_grouped(X, W.expand(3, N, K).contiguous(), [3, 0, 5]) == K).all()
        assert t.device_status() == 0
        t.close()


@pytest.mark.parametrize("layout", ["NK", "KN"])
@pytest.mark.parametrize("M,N,K,few", [(8, 64, 4096, True), (8, 64, 16384, False), (64, 64, 131072, False), (1, 512, 32768, False),
                                       (16, 2048, 14336, True), (64, 4096, 4096, True), (64, 8192, 1024, False),
                                       (32, 28672, 256, False), (8, 28672, 256, True)])
def test_long_k_of_few_columns_is_cut_into_slices(h, layout, M, N, K, few):  # noqa: F811
    """One CTA's walk over all of K is not what a few columns wait for; a call without scratch has no slices to take."""
    from paper_2604_26666_b200 import binding as bd

    case = mk("few_long", M, N, K, op="gemm", layout=layout, out="f32")
    ins = small_int_inputs(case, 9, lo=-2, hi=2)
    c = h.get_config("gemm", 1, M, N, K, layout=layout, out_dtype=torch.float32)
    assert (c.schedule == 4) == few
    X, W = ins.X.cuda(), ins.W.cuda()
    want = (ins.X.float() @ (ins.W if layout == "KN" else ins.W.t()).float())  # (exact: integers below 2^24)
    assert torch.equal(h.gemm(X, W, layout=layout, out_dtype=torch.float32).cpu(), want)
    out = torch.empty(M, N, dtype=torch.float32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    assert bd.lib().fact_gemm(h._h, M, N, K, X.data_ptr(), K, W.data_ptr(), W.stride(0), bd.LAYOUTS[layout], out.data_ptr(), N,
                              1, None, None, 0, s) == 0
    assert torch.equal(out.cpu(), want) and h.device_status() == 0
