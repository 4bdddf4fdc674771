"""GPU parity of the bf16 grouped GEMM at the edges of its tiles: experts with 0, 1, 15, 16, 17,
127-130, 143-145, 255-257, 512 and 513 rows (row counts around the MMA's step of 16, around a TMEM
row half of 128 and around a tile of 256), in launches with tiles of at most 256 and of at most
128 rows, with expert widths that leave partial blocks of weight rows, one to many K blocks per
job and shared experts.  The route is given, every output is compared with the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import synth
from tests import layer_harness as H

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 15, 16, 17, 127, 128, 129, 130, 143, 144, 145, 255, 256, 257, 512, 513]
SMALL = [0, 1, 2, 16, 17, 127, 128, 129, 257] + [3] * 23

CASES = {
    # name: (rows per expert, d, m, shared experts)
    "one_k_block": (EDGES, 64, 64, 0),
    "partial_blocks": (EDGES, 320, 192, 0),
    "many_k_blocks": (EDGES, 640, 448, 1),
    "small_tiles": (SMALL, 192, 320, 0),
    "small_tiles_shared": (SMALL, 512, 64, 2),
}


@pytest.mark.parametrize("name", list(CASES))
def test_expert_tiles(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    rows, d, m, shared = CASES[name]
    rows = rows + [0] * (-len(rows) % 16)
    N, T = len(rows), sum(rows)
    cfg = synth.LayerConfig(name, T=T, d=d, N=N, k=1, m=m, n_shared=shared)
    L = synth.make_layer(cfg, seed=11)
    rng = np.random.default_rng(3)
    idx = np.repeat(np.arange(N, dtype=np.int32), rows)
    rng.shuffle(idx)
    gates = rng.uniform(0.1, 1.0, size=(T, 1)).astype(np.float32)
    idx = np.ascontiguousarray(idx.reshape(T, 1))
    f = H.gpu_forward(cfg, H.to_dev(L), torch.from_numpy(idx).cuda(), torch.from_numpy(gates).cuda())
    assert f["code"] == 0 and int(f["status"].item()) == 0
    assert np.array_equal(H.cpu(f["counts"]).numpy(), np.asarray(rows, np.int32))
    assert np.array_equal(H.cpu(f["perm"]).numpy(), oracle.permute(idx, N)["perm"])
    want = oracle.moe_forward(L["x"], idx, gates, L["W_gate"], L["W_up"], L["W_down"], L["Ws_gate"],
                              L["Ws_up"], L["Ws_down"])
    H.normwise_close(H.cpu(f["out"]).float().numpy(), want, H.OUT_TOL["bf16"])
