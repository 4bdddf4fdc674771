"""GPU parity of the fp32 grouped GEMM at the edges of its blocks: both block sizes (32 x 64
once they fill the GPU five times), K blocks with a remainder, an expert width that is no multiple of 4
(unaligned rows, copied 4 bytes at a time), a last column block of one column, shared experts and
experts without any row.  Compared in full with the oracle, tolerances of ``layer_harness``."""
import pytest
import torch

from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import synth
from tests.test_gpu_layer import _full_layer_check

pytestmark = pytest.mark.gpu

CASES = {
    "ragged_width": dict(T=65, d=68, N=5, k=2, m=33),
    "one_column_over": dict(T=129, d=132, N=64, k=1, m=65, n_shared=1),
    "empty_experts": dict(T=3, d=4, N=200, k=2, m=31),
    "large_blocks": dict(T=2051, d=196, N=12, k=8, m=260, n_shared=2),
    "large_blocks_ragged": dict(T=2700, d=256, N=3, k=3, m=129),
}


@pytest.mark.parametrize("name", list(CASES))
def test_fp32_grouped_gemm_tiles(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    _full_layer_check(synth.LayerConfig(name, dtype="fp32", **CASES[name]))
