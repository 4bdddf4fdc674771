"""A layer whose routed and shared rows together pass 2^31 (the shared experts' rows follow the
routed ones in H and Y): 2^20 tokens of 4 columns, top-8 of 8 experts and 2045 shared experts of
width 1, in fp32.  The first and last tokens and a sample of the others against the oracle.  More
rows than 32 bits count are refused."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import build
from paper_2606_00395_gb300 import synth
from tests import layer_harness as H


@pytest.mark.gpu
def test_rows_past_2_to_the_31():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    cfg = synth.LayerConfig("rows", T=1 << 20, d=4, N=8, k=8, m=1, n_shared=2045, dtype="fp32")
    assert cfg.T * (cfg.k + cfg.n_shared) > 2**31 > cfg.T * cfg.n_shared
    dm = H.dims_of(cfg)
    if torch.cuda.mem_get_info()[0] < 1.2 * B.pr2_moe_workspace_bytes(dm):
        pytest.skip("not enough device memory")
    L = synth.make_layer(cfg, seed=9)
    rng = np.random.default_rng(9)
    idx = np.argsort(rng.random((cfg.T, cfg.N)), axis=1)[:, :cfg.k].astype(np.int32)
    gates = rng.uniform(0.1, 1.0, size=(cfg.T, cfg.k)).astype(np.float32)
    f = H.gpu_forward(cfg, H.to_dev(L), torch.from_numpy(idx).cuda(), torch.from_numpy(gates).cuda())
    torch.cuda.synchronize()
    assert f["code"] == 0 and int(f["status"].item()) == 0
    toks = np.unique(np.concatenate([rng.choice(cfg.T, size=300, replace=False), [0, cfg.T - 1]]))
    want = oracle.moe_forward(L["x"][torch.from_numpy(toks)], idx[toks], gates[toks], L["W_gate"], L["W_up"],
                              L["W_down"], L["Ws_gate"], L["Ws_up"], L["Ws_down"])
    H.normwise_close(H.cpu(f["out"]).numpy()[toks], want, H.OUT_TOL["fp32"])


def test_row_numbers_beyond_32_bits_are_refused():
    """On the host, whatever the workspace, before any CUDA call."""
    build.build()
    dm = B.dims(1 << 20, 4, 8, 8, 1, 4095, "fp32")
    fake = ctypes.c_void_p(256)
    code = B.load().pr2_moe_forward(ctypes.byref(dm), *[fake] * 10, None, None, fake, 1 << 40, None, None, None)
    assert code == 2  # PR2_ERR_UNSUPPORTED
