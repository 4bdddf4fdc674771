"""GPU parity of the predictive loss where its rows are finished by warps (N = 128, clusters of 4
and 8 CTAs): batches that end inside a CTA's rows, both objectives, teacher rows with zero
entries and invalid cache positions.  Bounds as in the predictive-loss parity tests."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import synth
from tests.test_gpu_predictor import _check, _gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("delta", [False, True])
@pytest.mark.parametrize("Tc", [1, 31, 640, 2433, 4000])
def test_loss_rows_by_warps(Tc, delta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    cfg = synth.LayerConfig("rows", T=Tc + 5, d=512, N=128, k=8, m=64)
    c = synth.make_loss_inputs(cfg.N, cfg.d, Tc, Tc + 5, seed=Tc)
    c["rho"][::3, 7::11] = 0.0
    c["rho"] /= c["rho"].sum(1, keepdim=True)
    g = _gpu(cfg, c, delta=delta)
    _check(cfg, c, g, delta=delta)
    if Tc < 31:
        return
    pos = c["pos"].numpy().copy()
    pos[[0, Tc // 2, Tc - 1]] = [-1, Tc + 5, 1 << 30]
    g = _gpu(cfg, c, delta=delta, pos=pos)
    ref = oracle.predictor_loss(c["h_old"], c["p_old"], c["W_pred"], c["rho"], pos=pos, delta=delta)
    assert g["status"] == B.PR2_STATUS_BAD_INDEX
    assert np.all(g["kl"][[0, Tc // 2, Tc - 1]] == 0)
    assert np.max(np.abs(g["grad"] - ref["grad"])) <= 1e-2 * np.max(np.abs(ref["grad"]))
    assert abs(g["loss"] - ref["loss"]) <= 1e-4 * abs(ref["loss"]) + 1e-7
