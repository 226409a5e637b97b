"""Whose memory the binding's scratch is, with the CUDA calls faked: of the
call's stream when that is not the current one (a tensor would go back to the
current stream's pool, and to its next allocation, before the call has run)."""
import pytest
import torch

import paper_1512_06473_gb300 as q


@pytest.fixture
def cuda(monkeypatch):
    log = []

    def alloc(size, device=None, stream=None):
        log.append(("alloc", size, stream))
        return 1000

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    monkeypatch.setattr(torch.cuda, "caching_allocator_delete", lambda p: log.append(("free", p)))
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(q, "_raw_stream", lambda device: 5)
    return log


class Stream:
    cuda_stream = 7


@pytest.mark.parametrize("stream", [7, Stream(), 0], ids=["handle", "object", "default stream"])
def test_another_stream_gives_its_own_memory(cuda, stream):
    ws, have = q._workspace(300, torch.device("cuda", 0), None, stream)
    assert have == 300 and ws.data_ptr() % 256 == 0
    (_, size, of), = cuda
    assert of == (0 if stream == 0 else 7)
    assert 1000 <= ws.data_ptr() and ws.data_ptr() + 300 <= 1000 + size
    del ws
    assert cuda[1:] == [("free", 1000)]


@pytest.mark.parametrize("stream", [None, 5])
def test_the_current_stream_gives_a_tensor(cuda, stream):
    ws, have = q._workspace(300, torch.device("cpu"), None, stream)
    assert isinstance(ws, torch.Tensor) and have >= 300 and not cuda


def test_the_callers_workspace_stays(cuda):
    mine = torch.empty(512, dtype=torch.uint8)
    assert q._workspace(300, torch.device("cpu"), mine, 7) == (mine, 512)
    assert q._workspace(0, torch.device("cpu"), mine, 7) == (None, 0) and not cuda
