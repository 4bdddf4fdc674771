"""The optional outputs of the layer forward are outputs only: another stream that writes to a
`perm` or `counts` buffer while the call runs (two streams given one buffer) mixes up that buffer
and leaves the layer's output alone."""
import numpy as np
import pytest
import torch

from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import synth
from tests import layer_harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,dtype", [(16384, "bf16"), (4096, "fp32")])
def test_output_buffers_written_by_another_stream(T, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    cfg = synth.LayerConfig("shared", T=T, d=512, N=32, k=8, m=512, dtype=dtype)
    L = H.to_dev(synth.make_layer(cfg, seed=5))
    rng = np.random.default_rng(5)
    idx = torch.from_numpy(np.argsort(rng.random((T, cfg.N)), axis=1)[:, :cfg.k].astype(np.int32)).cuda()
    gates = torch.from_numpy(rng.uniform(0.1, 1.0, size=(T, cfg.k)).astype(np.float32)).cuda()
    want = H.gpu_forward(cfg, L, idx, gates)["out"]

    dm = H.dims_of(cfg)
    out, ws = torch.empty_like(want), B.alloc_workspace(dm)
    perm = torch.empty(T * cfg.k, dtype=torch.int32, device="cuda")
    counts = torch.empty(cfg.N, dtype=torch.int32, device="cuda")
    # slot 0 everywhere: in range wherever it is read.  Copies, because no block of another kernel
    # fits beside the GEMM's.
    zeros = torch.zeros(T * cfg.k, dtype=torch.int32).pin_memory()
    dispatched, other = torch.cuda.Event(), torch.cuda.Stream()
    dispatched.record()  # creates the event that the call records again
    torch.cuda.synchronize()
    events = B.StageEvents(dispatched=dispatched.cuda_event)
    code = B.pr2_moe_forward(dm, L["x"], idx, gates, L["W_gate"], L["W_up"], L["W_down"], None, None,
                             None, out, counts, perm, ws, events=events)
    other.wait_event(dispatched)
    with torch.cuda.stream(other):
        perm.copy_(zeros, non_blocking=True)
        counts.copy_(zeros[:cfg.N], non_blocking=True)
    torch.cuda.synchronize()
    assert code == 0
    assert torch.equal(out, want)
