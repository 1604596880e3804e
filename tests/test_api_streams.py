"""CPU: a readout writes a fresh tensor on the state's own stream.  Torch's allocator
may give it the memory of a freed tensor that work queued on the current stream
still reads, so the write has to come after that work.  Torch's device calls and
the library's are stand-ins that record their order."""

import types

import pytest
import torch

from paper_1112_1805_gb300 import api
from paper_1112_1805_gb300 import binding as B


class Stream:
    def __init__(self, name, log, idle=False):
        self.name, self.log, self.idle = name, log, idle

    def query(self):
        return self.idle

    def wait_stream(self, other):
        self.log.append(f"{self.name} waits for {other.name}")

    def synchronize(self):
        self.log.append(f"{self.name} ends")


@pytest.mark.parametrize("cls,prefix", [(api.ShearletSegmenter, "seg"), (api.TVSegmenter, "tv"), (api.NLSegmenter, "nl"),
                                        (api._BorrowedState, "seg")])
@pytest.mark.parametrize("idle", [False, True])
def test_readouts_come_after_the_current_stream(monkeypatch, cls, prefix, idle):
    log = []
    current = Stream("current", log, idle)
    cuda = types.SimpleNamespace(current_stream=lambda: current, is_current_stream_capturing=lambda: False)
    fake = types.SimpleNamespace(cuda=cuda, float32=torch.float32, int32=torch.int32, float64=torch.float64,
                                 tensor=torch.tensor, empty=lambda shape, dtype, device: torch.empty(shape, dtype=dtype))
    monkeypatch.setattr(api, "torch", fake)
    monkeypatch.setattr(B, f"{prefix}_admm_get", lambda *a: log.append("get"))
    monkeypatch.setattr(B, f"{prefix}_admm_sync", lambda h: log.append("sync"))
    st = cls.__new__(cls)
    st.handle, st.K, st.C, st.H, st.W, st.eta, st.m = 1, 3, 1, 8, 8, 5, 10
    if cls is not api._BorrowedState:
        st.stream = Stream("own", log)
    assert tuple(st.get(B.SEG_W).shape) == (3, 8, 8)
    st.handle = None
    before = [] if idle else (["current ends"] if cls is api._BorrowedState else ["own waits for current"])
    assert log == before + ["get", "sync"]
