"""CPU: a readout writes a fresh tensor on the state's own stream.  Torch's allocator
may give it the memory of a freed tensor that work queued on the current stream
still reads, so the library is told that stream and orders the write after it
(tests/test_state_memory_host.py checks that it does).  Torch's device calls and the
library's are stand-ins."""

import types

import pytest
import torch

from paper_1112_1805_gb300 import api
from paper_1112_1805_gb300 import binding as B


@pytest.mark.parametrize("cls,prefix", [(api.ShearletSegmenter, "seg"), (api.TVSegmenter, "tv"), (api.NLSegmenter, "nl"),
                                        (api._BorrowedState, "seg")])
def test_readouts_name_the_current_stream(monkeypatch, cls, prefix):
    log = []
    cuda = types.SimpleNamespace(current_device=lambda: 3)
    raw = types.SimpleNamespace(_cuda_getCurrentRawStream=lambda device: 1231 + device)
    fake = types.SimpleNamespace(cuda=cuda, _C=raw, float32=torch.float32, int32=torch.int32, float64=torch.float64,
                                 tensor=torch.tensor, empty=lambda shape, dtype, device: torch.empty(shape, dtype=dtype))
    monkeypatch.setattr(api, "torch", fake)
    for name in ("get", "read", "sync"):
        monkeypatch.setattr(B, f"{prefix}_admm_{name}", lambda *a, name=name: log.append((name,) + a))
    st = cls.__new__(cls)
    st.handle, st.K, st.C, st.H, st.W, st.eta, st.m = 7, 3, 1, 8, 8, 5, 10
    out = st.get(B.SEG_W)
    st.handle = None
    assert tuple(out.shape) == (3, 8, 8) and log == [("read", 7, B.SEG_W, out.data_ptr(), 1234)]
