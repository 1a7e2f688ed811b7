"""The extension's marshalling against the ctypes marshalling (a call that names its stream): the same bits from every
method, the same errors for wrong arguments, and the library's kept choices follow the tuner's table."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    from paper_2604_26666_b200.binding import Handle
    hd = Handle(0)
    assert hd._bind.__name__ == "_fact_bind"  # (the tree's extension is current and in use)
    yield hd
    hd.close()


def rnd(*shape, scale=1.0, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn(shape, generator=g, device="cuda") * scale).to(torch.bfloat16)


def calls(h):
    x, w, wk = rnd(130, 264), rnd(320, 264, scale=0.05), rnd(264, 320, scale=0.05)
    b, r = rnd(320), rnd(130, 320)
    x8, w8 = rnd(96, 256).to(torch.float8_e4m3fn), rnd(160, 256).to(torch.float8_e4m3fn)
    q, k = rnd(2, 70, 4, 64), rnd(2, 70, 2, 64)
    wide = rnd(130, 304)[:, 8:272]  # a view with a leading dimension of its own
    yield lambda **kw: h.gemm(x, wk, **kw)
    yield lambda **kw: h.gemm(wide, w, layout="NK", out_dtype=torch.float32, **kw)
    yield lambda **kw: h.gemm_batched(rnd(3, 64, 128), rnd(3, 128, 72), **kw)
    yield lambda **kw: h.gemm_splitk(rnd(64, 8192), rnd(8192, 64, seed=1), **kw)  # (wants a workspace)
    yield lambda **kw: h.linear(x, w, bias=b, residual=r, epilogue="BIAS_RESIDUAL", **kw)
    yield lambda **kw: h.linear(x[:1], w, bias=b, epilogue="BIAS_GELU_TANH", **kw)
    yield lambda **kw: h.linear(torch.nn.Parameter(x, requires_grad=False), w, epilogue="SILU_GATE", **kw)
    yield lambda **kw: h.linear_fp8(x8, w8, 0.5, bias=b[:160], epilogue="BIAS", **kw)
    yield lambda **kw: h.linear_fp8(x8.view(torch.uint8), w8.view(torch.uint8), 2, **kw)
    yield lambda **kw: h.linear_grouped(x, rnd(3, 96, 264, scale=0.05), [50, 0, 80], **kw)
    yield lambda **kw: h.linear_grouped_fp8(x8, torch.stack([w8, w8]), [40, 56], 0.25, **kw)
    yield lambda **kw: h.attention(q, k, k, causal=True, **kw)
    yield lambda **kw: h.attention(q[:, :1], k, k, causal=False, scale=0.3, **kw)
    yield lambda **kw: h.norm(rnd(9, 768), rnd(768), rnd(768), kind="layer", **kw)
    yield lambda **kw: h.norm(rnd(9, 4096), rnd(4096), kind="rms", **kw)


def test_same_bits_as_the_ctypes_path(h):
    for n, f in enumerate(calls(h)):
        want = f(stream=torch.cuda.current_stream())
        for out in (None, torch.full_like(want, 7.0)):
            got = f(out=out)
            assert out is None or got is out
            assert got.dtype == want.dtype and torch.equal(got, want), n
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            got = f()
        torch.cuda.current_stream().wait_stream(side)
        assert torch.equal(got, want), n
    assert h.device_status() == 0


def test_wrong_arguments_raise_what_they_raised(h):
    from paper_2604_26666_b200.binding import FactError

    x, w = rnd(64, 128), rnd(96, 128)
    launches = h.launch_count()
    with pytest.raises(ValueError, match="inner dimensions"):
        h.linear(x, rnd(96, 120))
    with pytest.raises(ValueError, match="shape"):
        h.gemm(x, w, layout="NK", out=torch.empty(32, 96, dtype=torch.bfloat16, device="cuda"))
    with pytest.raises(TypeError):
        h.gemm(x.float(), w, layout="NK")
    with pytest.raises(ValueError, match="devices"):
        h.gemm(x.cpu(), w, layout="NK")
    with pytest.raises(ValueError):
        h.gemm(x, w, layout="XX")
    with pytest.raises(KeyError):
        h.gemm(x, w, layout="NK", out_dtype=torch.float16)
    with pytest.raises(KeyError):
        h.linear(x, w, epilogue="NOPE")
    with pytest.raises(FactError):  # the epilogue needs a bias
        h.linear(x, w, epilogue="BIAS")
    with pytest.raises(FactError):  # rows that are not whole 16-byte pieces
        h.gemm(rnd(64, 130)[:, 1:129], w, layout="NK")
    with pytest.raises(ValueError):
        h.linear_grouped(x, rnd(2, 96, 128), [10, 20])
    with pytest.raises(FactError):
        h.attention(rnd(1, 4, 3, 64), rnd(1, 4, 2, 64), rnd(1, 4, 2, 64))
    # (None for what makes a call a grouped or an FP8 one does not make it another method's call)
    x8, w8 = x.to(torch.float8_e4m3fn), w.to(torch.float8_e4m3fn)
    for wrong in (lambda: h.linear_grouped(x, w, None), lambda: h.linear_fp8(x, w, None), lambda: h.linear_fp8(x8, w8, None),
                  lambda: h.linear_grouped_fp8(x, torch.stack([w, w]), [32, 32], None), lambda: h.linear_grouped_fp8(x8, w8, None)):
        with pytest.raises((TypeError, ValueError)):
            wrong()
    with pytest.raises((TypeError, ctypes.ArgumentError)):
        h.block_forward(ctypes.pointer(h.block_desc("gpt", 1, 64, 2, 2, 64, 128, {})), x)
    assert h.launch_count() == launches
    assert torch.isfinite(h.gemm(x, w, layout="NK").float()).all()


def test_a_call_that_fails_after_a_launch_is_raised_not_repeated(h):
    # the last linear layer of a block has misaligned weights: six kernels have been launched by then
    from paper_2604_26666_b200.binding import FactError

    C, ffn, T = 128, 256, 96
    x = rnd(T, C)
    w = {"norm1_gamma": rnd(C), "norm2_gamma": rnd(C), "wqkv": rnd(3 * C, C), "wo": rnd(C, C), "w1": rnd(ffn, C), "b1": rnd(ffn)}
    good = h.block_desc("gpt", 1, T, 2, 2, 64, ffn, dict(w, w2=rnd(C, ffn)))
    bad = h.block_desc("gpt", 1, T, 2, 2, 64, ffn, dict(w, w2=rnd(C * ffn + 1)[1:].view(C, ffn)))
    h.block_forward(good, x)  # (the workspace has its size now)
    n = h.launch_count()
    h.block_forward(good, x)
    seven = h.launch_count() - n
    with pytest.raises(FactError, match="fact_block_forward"):
        h.block_forward(bad, x)
    assert h.launch_count() - n == 2 * seven - 1
    assert torch.isfinite(h.block_forward(good, x).float()).all() and h.device_status() == 0


def test_kept_choices_follow_the_table(h, tmp_path):
    M, N, K = 192, 256, 320
    x, w = rnd(M, K), rnd(N, K, scale=0.05)
    before, first = h.get_config("gemm", 1, M, N, K, layout="NK").as_dict(), h.gemm(x, w, layout="NK")
    other = 64 if before["tile_n"] != 64 else 128
    path = tmp_path / "table.txt"
    path.write_text(f"0 0 1 0 1 {M} {N} {K} | 128 {other} 64 4 1 1 1 2 1\n")
    h.tune_cache_load(str(path))
    assert h.get_config("gemm", 1, M, N, K, layout="NK").tile_n == other != before["tile_n"]
    assert torch.equal(h.gemm(x, w, layout="NK"), first)
