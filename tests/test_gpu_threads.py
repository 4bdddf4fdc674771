"""Calls of different layers from several host threads at once, each with its own stream and
buffers: no call refuses another's launch, and each gives the bits it gives alone.  The layers
differ in the number of experts, which sets the shared memory of the dispatch and routing kernels;
the binding's calls run without the interpreter lock, so the launches do interleave."""
import threading

import numpy as np
import pytest
import torch

from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import synth
from tests import layer_harness as H

pytestmark = pytest.mark.gpu


def _calls(kind, T, N, k, dtype):
    """A function that issues one call on a stream, and the tensors that it writes."""
    cfg = synth.LayerConfig("threads", T=T, d=64, N=N, k=k, m=64, dtype=dtype)
    L = H.to_dev(synth.make_layer(cfg, seed=N))
    dm = H.dims_of(cfg)
    rng = np.random.default_rng(N)
    idx = torch.from_numpy(np.argsort(rng.random((T, N)), axis=1)[:, :k].astype(np.int32)).cuda()
    gates = torch.full((T, k), 0.25, device="cuda")
    out, ws = torch.empty_like(L["x"]), B.alloc_workspace(dm)
    experts = (L["W_gate"], L["W_up"], L["W_down"], None, None, None, out)
    if kind == "forward":
        return lambda s: B.pr2_moe_forward(dm, L["x"], idx, gates, *experts, workspace=ws, stream=s), [out]
    if kind == "replay":
        return (lambda s: B.pr2_route_replay(dm, L["x"], L["W_router"], idx, gates, stream=s)), [gates]
    return (lambda s: B.pr2_moe_rollout_forward(dm, L["x"], L["W_router"], L["W_pred"], idx, gates, None,
                                                None, *experts, workspace=ws, stream=s)), [out, idx, gates]


@pytest.mark.parametrize("kind,T,k,dtype,Ns,n", [
    ("forward", 64, 8, "fp32", (16, 256), 8000), ("forward", 64, 8, "bf16", (16, 256), 8000),
    ("forward", 25000, 4, "fp32", (16, 256), 3000), ("rollout", 40, 8, "bf16", (144, 256), 8000),
    ("replay", 300, 8, "bf16", (144, 256), 8000), ("replay", 20000, 4, "bf16", (16, 64), 3000)])
def test_layers_from_two_threads(kind, T, k, dtype, Ns, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    sides = [_calls(kind, T, N, k, dtype) for N in Ns]
    want = []
    for call, outs in sides:
        B.check(call(None))
        torch.cuda.synchronize()
        want.append([o.clone() for o in outs])
    codes = [[], []]
    start = threading.Barrier(2)

    def work(i):
        torch.zeros(1, device="cuda")  # the device's context is current in this thread
        stream = torch.cuda.Stream()
        start.wait()
        codes[i] = [sides[i][0](stream) for _ in range(n)]
        stream.synchronize()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert [sum(c != 0 for c in side) for side in codes] == [0, 0]
    for (_, outs), ref in zip(sides, want):
        assert all(torch.equal(o, r) for o, r in zip(outs, ref))


@pytest.mark.parametrize("kind", ["replay", "rollout"])
def test_first_call_of_a_host_thread(kind):
    """A thread whose first CUDA work is a routing call, on a stream that another thread made."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    call, outs = _calls(kind, 40, 16, 4, "bf16")
    B.check(call(None))
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    want = [o.clone() for o in outs]
    torch.cuda.synchronize()
    codes = []
    thread = threading.Thread(target=lambda: codes.append(call(stream)))
    thread.start()
    thread.join()
    stream.synchronize()
    assert codes == [0]
    assert all(torch.equal(o, w) for o, w in zip(outs, want))
