"""Row normalisation at the edges of its variants (a warp or a CTA per row; one, two or four chunks of 8 values per thread)
against the FP64 oracle, under the BF16 gates of the block tests' norms."""
import pytest
import torch

from oracle import block as ob
from tests.test_block_gpu import DEV, rnd
from tests.helpers import to_f64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    from paper_2604_26666_b200.binding import Handle
    hd = Handle(0)
    yield hd
    hd.close()


@pytest.mark.parametrize("kind", ["layer", "rms"])
@pytest.mark.parametrize("M,C", [(1, 8), (9, 256), (3, 264), (2048, 512), (2049, 512), (5, 1024), (1, 1032), (7, 2048), (3, 2056),
                                 (130, 4096), (2, 4104), (5, 8192)])
def test_norm_variants(h, kind, M, C):
    x, g, b = rnd((M, C), 41) * 3 + 0.5, 1 + rnd((C,), 42) * 0.1, rnd((C,), 43)
    x, g, b = (t.to(torch.bfloat16) for t in (x.float(), g.float(), b.float()))
    wide = torch.full((M, C + 8), -7.0, dtype=torch.bfloat16, device=DEV)
    h.norm(x.to(DEV), g.to(DEV), b.to(DEV) if kind == "layer" else None, kind=kind, out=wide[:, :C])
    torch.cuda.synchronize()
    xf, gf = to_f64(x), to_f64(g)
    ref = torch.from_numpy(ob.layer_norm(xf, gf, to_f64(b), 1e-5) if kind == "layer" else ob.rms_norm(xf, gf, 1e-5))
    err = (wide[:, :C].cpu().double() - ref).abs()
    # one rounding to BF16 (2^-9 relative) and FP32 arithmetic over at most 8192 terms
    assert (err <= 2.0 ** -8 * ref.abs() + 1e-5).all()
    assert (wide[:, C:] == -7.0).all()


@pytest.mark.parametrize("kind", ["layer", "rms"])
@pytest.mark.parametrize("M,C", [(16384, 768), (16383, 768), (47663, 264), (24577, 512), (12288, 1024), (48000, 776)])
def test_streamed_rows(h, kind, M, C):
    """Many rows of 257 to 1024 values: a warp's rows, the last ones' ring slots, strided input and output; offsets or none."""
    g = torch.Generator(device=DEV).manual_seed(M + C)
    wide = torch.randn((M, C + 16), generator=g, device=DEV, dtype=torch.bfloat16) * 3 + 0.5
    x, gain = wide[:, 8:8 + C], 1 + torch.randn(C, generator=g, device=DEV, dtype=torch.bfloat16) * 0.1
    for beta in ([torch.randn(C, generator=g, device=DEV, dtype=torch.bfloat16), None] if kind == "layer" else [None]):
        out = torch.full((M, C + 8), -7.0, dtype=torch.bfloat16, device=DEV)
        h.norm(x, gain, beta, kind=kind, out=out[:, :C])
        torch.cuda.synchronize()
        assert h.device_status() == 0 and bool((out[:, C:] == -7.0).all())
        xd = x.double()
        if kind == "layer":
            xd = xd - xd.mean(1, keepdim=True)
        ref = xd / (xd.square().mean(1, keepdim=True) + 1e-5).sqrt() * gain.double() + (0.0 if beta is None else beta.double())
        # one rounding to BF16 (2^-9 relative) and FP32 arithmetic over at most 1024 terms
        assert bool(((out[:, :C].double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-5).all())
