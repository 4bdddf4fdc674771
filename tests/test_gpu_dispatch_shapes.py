"""GPU parity of dispatch in each of its launch shapes: one block (up to 1024 slots, any number of
experts), 256-slot blocks (up to 98304 slots) and 2048-slot blocks in one cooperative launch, and
three launches (numbers of experts that are no multiple of 4), at the edges between them and of
their last block, with invalid and repeated route entries.  Counts and permutation are bit equal to
the oracle's, the status word reports the invalid slots, and the layer output (which reads the tile
table) matches."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import synth
from tests import layer_harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,k,N,bad", [
    (1, 1, 16, False), (33, 3, 48, True), (256, 8, 128, False), (1024, 2, 256, True),
    (1025, 2, 16, False), (2048, 1, 32, True), (683, 3, 256, False),
    (131073, 1, 16, True), (16385, 8, 32, False), (40000, 4, 64, True)])
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_dispatch_shapes(T, k, N, bad, dtype):
    _check(T, k, N + 4 if dtype == "fp32" and T > 2048 else N, bad, dtype)


@pytest.mark.parametrize("T,k,N,bad,dtype", [
    # 1023, 1024 and 1025 slots: the last of one block, the first of several
    (341, 3, 16, True, "bf16"), (341, 3, 144, False, "bf16"), (341, 3, 256, True, "bf16"),
    (128, 8, 16, False, "bf16"), (128, 8, 144, True, "bf16"), (256, 4, 256, True, "bf16"),
    (205, 5, 16, True, "bf16"), (205, 5, 144, True, "bf16"), (205, 5, 256, False, "bf16"),
    (341, 3, 5, True, "fp32"), (128, 8, 251, True, "fp32"), (205, 5, 131, True, "fp32"),
    (64, 16, 33, True, "fp32"),
    # 98304 and 98305 slots: the last in blocks of 256, the first in blocks of 2048
    (12288, 8, 16, True, "bf16"), (24576, 4, 256, False, "bf16"),
    (19661, 5, 16, False, "bf16"), (19661, 5, 256, True, "bf16"), (98305, 1, 6, True, "fp32")])
def test_dispatch_edges(T, k, N, bad, dtype):
    _check(T, k, N, bad, dtype)


def _check(T, k, N, bad, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    d, m = 64, 64
    cfg = synth.LayerConfig("d", T=T, d=d, N=N, k=k, m=m, dtype=dtype)
    L = synth.make_layer(cfg, seed=2)
    rng = np.random.default_rng(T + k)
    idx = np.argsort(rng.random((T, N)), axis=1)[:, :k].astype(np.int32)
    if bad:
        rows = rng.choice(T, size=max(1, T // 7), replace=False)
        idx[rows[::2], rng.integers(0, k)] = N + 3
        idx[rows[1::2], k - 1] = idx[rows[1::2], 0] if k > 1 else -1
    gates = rng.uniform(0.1, 1.0, size=(T, k)).astype(np.float32)
    f = H.gpu_forward(cfg, H.to_dev(L), torch.from_numpy(idx).cuda(), torch.from_numpy(gates).cuda())
    operm = oracle.permute(idx, N)
    nvalid = int(operm["offsets"][-1])
    assert np.array_equal(H.cpu(f["counts"]).numpy(), operm["counts"])
    assert np.array_equal(H.cpu(f["perm"]).numpy()[:nvalid], operm["perm"][:nvalid])
    assert int(f["status"].item()) == (B.PR2_STATUS_BAD_INDEX if nvalid < T * k else 0)
    toks = np.unique(np.concatenate([rng.choice(T, size=min(T, 200), replace=False), [0, T - 1]]))
    want = oracle.moe_forward(L["x"][torch.from_numpy(toks)], idx[toks], gates[toks], L["W_gate"],
                              L["W_up"], L["W_down"], None, None, None)
    H.normwise_close(H.cpu(f["out"]).float().numpy()[toks], want, H.OUT_TOL[dtype])
