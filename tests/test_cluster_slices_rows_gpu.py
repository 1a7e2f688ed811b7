"""K slices as a cluster: where the rows of the output and the residual lie.  The kernel stores 16 columns at once where
they start on 32 bytes, 8 at a time elsewhere, and single elements in a ragged last group; it loads bias and residual 64
columns ahead.  Bit for bit on integer-valued inputs (exact sums), columns around the output untouched."""
import pytest
import torch

from tests.helpers import oracle_for, small_int_inputs
from tests.test_any_rows_gpu import run_into
from tests.test_gemm_gpu import h, mk  # noqa: F401

pytestmark = pytest.mark.gpu


# 128 columns a CTA (two groups of 64 fetched), 32 (half a group, eight slices: the second four added on), pairs; N one
# past a store, past a 64-column group, in the first group; rows on 32, 16, 4 and 2 bytes
@pytest.mark.parametrize("pair,slices,tile_n", [(1, 2, 256), (1, 8, 256), (2, 2, 128), (1, 2, 64)])
@pytest.mark.parametrize("out", ["bf16", "f32"])
@pytest.mark.parametrize("epi", ["NONE", "BIAS_RESIDUAL"])
@pytest.mark.parametrize("N,ld,off", [(464, 464, 0), (465, 472, 8), (321, 322, 2), (77, 79, 1), (9, 9, 3)])
def test_rows_of_a_cluster_slice(h, epi, out, pair, slices, tile_n, N, ld, off):  # noqa: F811
    case = mk(f"kc_rows_{N}_{epi}", 197, N, 1096, epilogue=epi, layout="NK", out=out)
    ins = small_int_inputs(case, 17, lo=-2, hi=2)
    ref = torch.from_numpy(oracle_for(ins, case))
    got, intact = run_into(h, case, ins, ld, off,
                           {"cta_group": pair, "tile_n": tile_n, "split_k": slices, "schedule": 3})
    assert intact
    assert torch.equal(got.cpu().double(), ref.to(got.dtype).double())
