"""GPU parity of predict routing where its rows are finished by warps (N = 128 in clusters of 4 and
8 CTAs): batches that end inside a CTA's rows, in its first and last row and in a tile of few
rows (whose dead rows are not exchanged), every k, ties within and across the lanes' four experts
(duplicated router rows: the lower expert first), with and without the logits and the
renormalisation.  Routes, gates and logits against the oracle, tolerances of ``layer_harness``."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import synth
from tests import layer_harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,k,flags,logits", [
    (1, 8, 0, True), (15, 1, 0, True), (17, 3, B.PR2_F_NORMALIZE_TOPK, True), (128, 8, 0, False),
    (129, 5, 0, True), (2430, 8, B.PR2_F_NORMALIZE_TOPK, True), (2433, 2, 0, False),
    (4033, 8, 0, True), (4095, 4, 0, True)])
def test_predict_rows_by_warps(T, k, flags, logits):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    cfg = synth.LayerConfig("rows", T=T, d=512, N=128, k=k, m=64)
    L = synth.make_layer(cfg, seed=6)
    g = H.gpu_predict(cfg, H.to_dev(L), logits=logits, flags=flags)
    orc = oracle.route_predict(L["x"], L["W_router"], L["W_pred"], k)
    idx = H.cpu(g["idx"]).numpy()
    H.check_routes(orc, idx)
    want = np.take_along_axis(orc["probs"], idx, 1)
    if flags:
        want = want / want.sum(1, keepdims=True)
    H.rowwise_close(H.cpu(g["gates"]).numpy(), want)
    if logits:
        H.rowwise_close(H.cpu(g["logits"]).numpy(), orc["logits"])
    assert int(g["status"].item()) == 0


@pytest.mark.parametrize("T", [40, 3000])
def test_equal_logits_take_the_lower_expert(T):
    """Experts 8 j, 8 j + 3 and 8 j + 5 share their router and predictor rows: their logits are
    the same bits, and they have to come out in index order."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    cfg = synth.LayerConfig("equal", T=T, d=256, N=128, k=8, m=64)
    L = synth.make_layer(cfg, seed=7)
    for W in (L["W_router"], L["W_pred"]):
        W[3::8] = W[0::8]
        W[5::8] = W[0::8]
    idx = H.cpu(H.gpu_predict(cfg, H.to_dev(L))["idx"]).numpy()
    for row in idx:
        where = {int(e): s for s, e in enumerate(row)}
        for e, s in where.items():
            if e % 8 == 3:
                assert where.get(e - 3, 99) == s - 1, row
            if e % 8 == 5:
                assert where.get(e - 2, 99) == s - 1, row
