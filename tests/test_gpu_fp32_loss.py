"""GPU parity of the fp32 predictive loss and its gradient where the kernels' blocks end: expert
counts that are no multiple of 8 or 32, columns that end inside a block of 32, tokens around the
gradient's blocks of 64, one and four tokens per warp, both objectives.  Bounds as in the
predictive-loss parity tests."""
import pytest
import torch

from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import synth
from tests.test_gpu_predictor import _check, _gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("delta", [False, True])
@pytest.mark.parametrize("T,N,d", [(1, 2, 4), (63, 7, 36), (65, 33, 132), (128, 8, 32),
                                   (129, 50, 500), (515, 64, 260), (1021, 200, 84)])
def test_fp32_loss(T, N, d, delta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    cfg = synth.LayerConfig("fp32", T=T + 5, d=d, N=N, k=1, m=64, dtype="fp32")
    c = synth.make_loss_inputs(N, d, T, T + 5, seed=T, dtype="fp32")
    _check(cfg, c, _gpu(cfg, c, delta=delta), delta=delta)
