"""The binding asks torch's C layer for the current stream only while CUDA is initialised in this
very process: before that, and in a process forked from one that used CUDA, torch's own call decides
(it initialises CUDA or raises).  torch's calls are stood in for, so no GPU is needed."""
import types

import pytest
import torch

from paper_2606_00395_gb300 import binding as B


def test_forked_process_asks_torch(monkeypatch):
    live = types.SimpleNamespace(on=True)

    def current_stream():
        if not live.on:
            raise RuntimeError("Cannot re-initialize CUDA in forked subprocess")
        return types.SimpleNamespace(cuda_stream=7)

    monkeypatch.setattr(torch.cuda, "current_stream", current_stream)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: live.on)
    monkeypatch.setattr(B, "_get_device", lambda: 3)
    monkeypatch.setattr(B, "_raw_stream", lambda dev: {3: 7}[dev])
    assert [B._s(None), B._s(None), B._s(5)] == [7, 7, 5]
    live.on = False  # what is_initialized says after a fork
    with pytest.raises(RuntimeError, match="forked"):
        B._s(None)
