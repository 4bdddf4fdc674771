"""A bounded wait that runs out in the rollout layer's routing kernel leaves the route unwritten and
sets the timeout bit.  What runs behind it then trusts neither the route nor its histograms: dispatch
(called here by itself, on a route and histograms of arbitrary bits) writes nothing, and without a
status word of the caller's the workspace's own is cleared in front of the routing kernel, so that
its bit is still there when dispatch, the GEMM and the combine look."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2606_00395_gb300 import binding as B
from paper_2606_00395_gb300 import synth
from tests import layer_harness as H

pytestmark = pytest.mark.gpu

P = ctypes.c_void_p


class DispatchArgs(ctypes.Structure):
    """``pr2::DispatchArgs`` of csrc/pr2_internal.h."""

    _fields_ = [("idx", P), ("T", ctypes.c_int64), ("k", ctypes.c_int), ("N", ctypes.c_int),
                ("n_shared", ctypes.c_int), ("blk_hist", P), ("counts", P), ("offsets", P), ("perm", P),
                ("inv", P), ("tiles", P), ("num_tiles", P), ("status", P), ("sync_ctr", P), ("ready", P),
                ("tile_rows", ctypes.c_int)]


def _dispatch_from_hist(idx, hist, N, status):
    T, k = idx.shape
    max_tiles = T * k // 128 + N + 1
    out = {n: torch.full((s,), -7, dtype=torch.int32, device="cuda")
           for n, s in dict(counts=N, offsets=N + 1, perm=T * k, inv=T * k, tiles=4 * max_tiles,
                            num_tiles=1, ready=max_tiles).items()}
    st = torch.tensor([status], dtype=torch.int32, device="cuda")
    fn = B.load()._ZN3pr225launch_dispatch_from_histERKNS_12DispatchArgsEPKiiP11CUstream_st
    fn.argtypes, fn.restype = [ctypes.POINTER(DispatchArgs), P, ctypes.c_int, P], ctypes.c_int
    args = DispatchArgs(idx=idx.data_ptr(), T=T, k=k, N=N, n_shared=0, status=st.data_ptr(), tile_rows=128,
                        **{n: t.data_ptr() for n, t in out.items()})
    split = hist.shape[0] // ((T + 127) // 128)
    assert fn(ctypes.byref(args), hist.data_ptr(), split, torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    return {n: t.cpu().numpy() for n, t in out.items()}


@pytest.mark.parametrize("T,k,N", [(1, 1, 16), (300, 8, 128), (1000, 6, 256)])
def test_dispatch_behind_a_routing_timeout(T, k, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(N)
    bits = lambda *s: torch.from_numpy(rng.integers(-2**31, 2**31, size=s).astype(np.int32)).cuda()  # noqa: E731
    tiles = (T + 127) // 128
    out = _dispatch_from_hist(bits(T, k), bits(tiles * 2, N), N, B.PR2_STATUS_TIMEOUT)
    assert all(np.all(v == -7) for v in out.values())

    # without the bit: the valid slots are placed, one that names no expert is not
    idx = np.argsort(rng.random((T, N)), axis=1)[:, :k].astype(np.int32)
    idx[T // 2, k - 1] = N
    idx[T - 1, 0] = -2**31
    hist = np.zeros((tiles, N), np.int32)
    for b in range(tiles):
        e = idx[128 * b:128 * b + 128].reshape(-1)
        hist[b] = np.bincount(e[(e >= 0) & (e < N)], minlength=N)
    out = _dispatch_from_hist(torch.from_numpy(idx).cuda(), torch.from_numpy(hist).cuda(), N, 0)
    ref = oracle.permute(idx, N)
    n = int(ref["offsets"][-1])
    assert np.array_equal(out["counts"], ref["counts"]) and np.array_equal(out["offsets"], ref["offsets"])
    assert np.array_equal(out["perm"][:n], ref["perm"][:n])
    assert np.array_equal(np.flatnonzero(out["inv"] == -1),
                          np.flatnonzero((idx.reshape(-1) < 0) | (idx.reshape(-1) >= N)))


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_own_status_word_is_cleared_before_routing(dtype):
    """The first node of the captured call is the memset of the workspace's status word."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load()
    cfg = synth.LayerConfig("status", T=40, d=64, N=16, k=4, m=64, dtype=dtype)
    L = H.to_dev(synth.make_layer(cfg, seed=1))
    dm = H.dims_of(cfg)
    idx, gates, _ = B.alloc_route(dm)
    out, ws = torch.empty_like(L["x"]), B.alloc_workspace(dm)

    def call(stream):
        return B.pr2_moe_rollout_forward(dm, L["x"], L["W_router"], L["W_pred"], idx, gates, None, None,
                                         L["W_gate"], L["W_up"], L["W_down"], None, None, None, out,
                                         workspace=ws, stream=stream)

    stream = torch.cuda.Stream()
    B.check(call(stream))
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    graph, node, n, kind = P(), P(), ctypes.c_size_t(1), ctypes.c_int(-1)
    s = P(stream.cuda_stream)
    relaxed, memset = 2, 2  # CU_STREAM_CAPTURE_MODE_RELAXED, CU_GRAPH_NODE_TYPE_MEMSET
    assert cu.cuStreamBeginCapture_v2(s, relaxed) == 0
    code = call(stream)
    assert cu.cuStreamEndCapture(s, ctypes.byref(graph)) == 0 and code == 0
    assert cu.cuGraphGetRootNodes(graph, ctypes.byref(node), ctypes.byref(n)) == 0 and n.value == 1
    assert cu.cuGraphNodeGetType(node, ctypes.byref(kind)) == 0 and kind.value == memset
    assert cu.cuGraphDestroy(graph) == 0
