"""The fp32 multi-layer rollout with T N no multiple of 4, so that the later layers' logits start at
any float of the caller's buffer: every layer runs and agrees with the oracle composition, for a
buffer that starts on 16 bytes; one that does not is refused before anything is written."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import synth
from tests import layer_harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,N,L", [(3, 5, 2), (37, 9, 4), (2, 7, 3)])
def test_fp32_layers_with_logits_at_any_float(T, N, L):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    cfg = synth.LayerConfig("slices", T=T, d=64, N=N, k=2, m=32, dtype="fp32")
    layers = [synth.make_layer(cfg, seed=70 + l) for l in range(L)]
    W = {n: torch.stack([w[n] for w in layers]).cuda()
         for n in ("W_router", "W_pred", "W_gate", "W_up", "W_down")}
    h0 = layers[0]["x"].cuda()
    dm = H.dims_of(cfg)
    ws = B.alloc_workspace(dm)
    idx = torch.full((L, T, 2), -1, dtype=torch.int32, device="cuda")
    gates = torch.zeros(L, T, 2, device="cuda")
    store = torch.zeros(L * T * N + 1, device="cuda")

    def call(h, logits):
        return B.pr2_rollout_layers(dm, L, h, W["W_router"], W["W_pred"], W["W_gate"], W["W_up"], W["W_down"],
                                    idx, gates, logits_old=logits, workspace=ws)

    h = h0.clone()
    assert call(h, store[1:]) == 1  # PR2_ERR_INVALID_ARG
    torch.cuda.synchronize()
    assert torch.equal(h, h0) and int(idx.max()) == -1
    assert call(h, store[:-1]) == 0
    torch.cuda.synchronize()
    logits = H.cpu(store[:-1]).numpy().reshape(L, T, N)
    x = layers[0]["x"]
    for l, w in enumerate(layers):  # each layer on the stream that the oracle's layers before it give
        ref = oracle.route_predict(x, w["W_router"], w["W_pred"], 2)
        H.check_routes(ref, H.cpu(idx[l]).numpy())
        H.rowwise_close(logits[l], ref["logits"])
        out = oracle.moe_forward(x, ref["idx"], ref["gates"], w["W_gate"], w["W_up"], w["W_down"])
        x = (x.double() + torch.from_numpy(np.asarray(out))).float()
    H.normwise_close(H.cpu(h).numpy(), x.numpy(), H.OUT_TOL["fp32"])
