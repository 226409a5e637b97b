"""Scratch where there is no room for the contraction's: the least sizes, and the
binding's way down to them (allocations faked)."""
import ctypes

import pytest
import torch

import paper_1512_06473_gb300 as q
from paper_1512_06473_gb300 import _lib


def size(query, *args):
    nb = ctypes.c_size_t()
    _lib.check(getattr(q.load(), query)(*args, ctypes.byref(nb)), query)
    return nb.value


def test_least_sizes_are_the_table_plans():
    conv = (32, 256, 28, 28, 512, 3, 3, 1, 1, 8, 128)
    table = q.conv_plan(*conv[:9], Csp=8, K=128)["algo"]
    for layout in (_lib.CODES_PACKED, _lib.CODES_CANONICAL):
        least = size("qcnn_conv_workspace_min", *conv, layout, 0, 0)
        assert least == size("qcnn_conv_workspace_size", *conv, layout, _lib.ALGO[table], 0)
        assert least < size("qcnn_conv_workspace_size", *conv, layout, 0, 0)
        for algo in ("contract", "fused"):  # asked for: no less will do
            args = (*conv, layout, _lib.ALGO[algo], 0)
            assert size("qcnn_conv_workspace_min", *args) == size("qcnn_conv_workspace_size", *args)
    fc = (64, 4096, 1000, 4, 32, 0)
    p = q.fc_plan(*fc[:5])
    assert size("qcnn_fc_workspace_min", *fc) == \
        -(-(p["splits"] // p["cluster"] * 64 * 1000 * 4) // 256) * 256
    small = (1, 64, 40, 4, 16, 0)
    assert size("qcnn_fc_workspace_min", *small) == size("qcnn_fc_workspace_size", *small)


def test_errors_are_those_of_the_sizes():
    lib, nb = q.load(), ctypes.c_size_t()
    assert lib.qcnn_fc_workspace_min(2, 10, 4, 4, 16, 0, ctypes.byref(nb)) == _lib.ERR_INVALID_ARG
    assert lib.qcnn_fc_workspace_min(2, 8, 4, 4, 16, 0, None) == _lib.ERR_INVALID_ARG
    assert lib.qcnn_conv_workspace_min(1, 8, 9, 9, 4, 3, 3, 2, 1, 4, 16, 0, 1, 0,
                                       ctypes.byref(nb)) == _lib.ERR_UNSUPPORTED
    assert lib.qcnn_net_workspace_min(None, 0, 1, 3, 9, 9, 0, ctypes.byref(nb)) == \
        _lib.ERR_INVALID_ARG


@pytest.mark.parametrize("room,least,got", [(1000, None, 1000), (500, 300, 300), (500, 0, 0)])
def test_no_room_for_the_full_size(monkeypatch, room, least, got):
    real = torch.empty

    def empty(n, **kw):
        if n > room:
            raise torch.cuda.OutOfMemoryError("no room")
        return real(n, **kw)

    monkeypatch.setattr(torch, "empty", empty)
    # (the host's allocator: a start off 256 bytes would ask for more)
    monkeypatch.setattr(torch.Tensor, "data_ptr", lambda t: 256)
    ws, n = q._workspace(1000, "cpu", None, None, None if least is None else (int, least))
    assert n == got and (ws is None) == (got == 0)


@pytest.mark.parametrize("least", [None, (int, 1000), (int, 800)])
def test_no_room_at_all(monkeypatch, least):
    def empty(n, **kw):
        raise torch.cuda.OutOfMemoryError("no room")

    monkeypatch.setattr(torch, "empty", empty)
    with pytest.raises(torch.cuda.OutOfMemoryError):
        q._workspace(1000, "cpu", None, None, least)


@pytest.mark.gpu
def test_calls_without_room_run_their_tables():
    g = torch.Generator(device="cuda").manual_seed(31)
    x = torch.randn((64, 256, 56, 56), generator=g, device="cuda")
    D = torch.randn((64, 64, 4), generator=g, device="cuda")
    c = torch.randint(0, 64, (64, 9, 64), generator=g, device="cuda", dtype=torch.uint8)
    packed = q.conv_pack_codes(c, 64, 3, 3)
    net = q.Net([q.ConvLayer(D, packed, None, 64, 3, 3, 1, 1, relu=False, packed=True)], (256, 56, 56))
    out, out2 = (torch.empty((64, 64, 56, 56), device="cuda") for _ in range(2))
    plan = q.conv_plan(64, 256, 56, 56, 64, 3, 3, 1, 1, 4, 64)["algo"]
    assert q.conv_route(64, 256, 56, 56, 64, 3, 3, 1, 1, 4, 64)["algo"] == "contract"
    want = q.conv_forward(x, D, packed, 3, 3, 1, 1, packed=True, Ct=64, algo=plan)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = torch.cuda.memory_reserved() + (64 << 20)
    try:
        torch.cuda.set_per_process_memory_fraction(
            room / torch.cuda.get_device_properties(0).total_memory)
        q.conv_forward(x, D, packed, 3, 3, 1, 1, packed=True, Ct=64, out=out)
        net.forward(x, out=out2)
        torch.cuda.synchronize()
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert torch.equal(out, want) and torch.equal(out2, want)
