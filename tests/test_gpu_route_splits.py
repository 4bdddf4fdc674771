"""GPU parity of bf16 routing in clusters of 8, 4, 2 and 1 CTAs with every kind of split: expert
counts that no cluster size divides into sixteens, numbers of K blocks that it does not divide, two,
four and eight experts per lane, partial rows exchanged in one round and in several or finished by
halves (N = 256), and batches that end inside the rows of a CTA.  Predict, replay (with invalid and
repeated slots) and the predictive loss against the oracle, tolerances of ``layer_harness`` and the
predictive-loss tests."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import synth
from tests import layer_harness as H
from tests.test_gpu_predictor import _check, _gpu

pytestmark = pytest.mark.gpu

# 1 .. 38 tiles of 128 tokens run in clusters of 4 or 8, 39 .. 76 in clusters of 2, 77 and more
# alone, from 153 on two to an SM where both fit
SHAPES = [(1, 16, 512, 4), (77, 80, 576, 8), (300, 144, 704, 8), (513, 256, 2112, 8),
          (900, 208, 320, 3), (2433, 240, 576, 8), (3001, 48, 832, 6), (4700, 256, 320, 8),
          (5003, 256, 192, 8), (5121, 176, 320, 5), (8200, 128, 448, 8), (9700, 64, 128, 8),
          (130, 64, 64, 2), (2000, 64, 1024, 6), (9800, 256, 128, 8), (10003, 224, 64, 8),
          (9999, 128, 192, 8), (12001, 32, 64, 4), (19500, 256, 64, 8),
          (1100, 128, 2048, 8)]


@pytest.mark.parametrize("T,N,d,k", SHAPES)
def test_predict_and_replay(T, N, d, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    flags = B.PR2_F_NORMALIZE_TOPK if T % 2 else 0
    cfg = synth.LayerConfig("splits", T=T, d=d, N=N, k=k, m=64)
    L = synth.make_layer(cfg, seed=T)
    Ld = H.to_dev(L)
    g = H.gpu_predict(cfg, Ld, flags=flags)
    orc = oracle.route_predict(L["x"], L["W_router"], L["W_pred"], k)
    idx = H.cpu(g["idx"]).numpy()
    H.check_routes(orc, idx)
    want = np.take_along_axis(orc["probs"], idx, 1)
    H.rowwise_close(H.cpu(g["gates"]).numpy(), want / want.sum(1, keepdims=True) if flags else want)
    H.rowwise_close(H.cpu(g["logits"]).numpy(), orc["logits"])
    assert int(g["status"].item()) == 0

    r = H.gpu_replay(cfg, Ld, Ld["W_router"], g["idx"], flags=flags)
    ref = oracle.route_replay(L["x"], L["W_router"], idx, normalize=bool(flags))
    H.rowwise_close(H.cpu(r["gates"]).numpy(), ref["gates"])
    H.rowwise_close(H.cpu(r["probs"]).numpy(), ref["probs"])
    assert int(r["status"].item()) == 0
    idx = idx.copy()
    idx[0, 0], idx[T // 2, k - 1], idx[T - 1, 1] = -1, N, idx[T - 1, 0]
    r = H.gpu_replay(cfg, Ld, Ld["W_router"], torch.from_numpy(idx).cuda(), flags=flags)
    ref = oracle.route_replay(L["x"], L["W_router"], idx, normalize=bool(flags))
    H.rowwise_close(H.cpu(r["gates"]).numpy(), ref["gates"])
    assert int(r["status"].item()) == B.PR2_STATUS_BAD_INDEX


@pytest.mark.parametrize("T,N,d,k", SHAPES)
def test_loss(T, N, d, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    cfg = synth.LayerConfig("splits", T=T + 5, d=d, N=N, k=k, m=64)
    c = synth.make_loss_inputs(N, d, T, T + 5, seed=T)
    c["rho"][::3, 7::11] = 0.0
    c["rho"] /= c["rho"].sum(1, keepdim=True)
    for delta in (False, True):
        _check(cfg, c, _gpu(cfg, c, delta=delta), delta=delta)
