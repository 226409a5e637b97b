"""Calls on another stream than the current one (``stream=``): their scratch is
not the next allocation of the current stream while they are still to run.

Each call is queued behind a spin on its stream, then as many bytes as its
scratch has are allocated and filled on the current stream: a block shared by
both would be written by the call's kernels afterwards."""
import ctypes

import pytest
import torch

import paper_1512_06473_gb300 as q

pytestmark = pytest.mark.gpu


def _calls():
    g = torch.Generator(device="cuda").manual_seed(3)

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    def codes(*shape):
        return torch.randint(0, 16, shape, generator=g, device="cuda", dtype=torch.uint8)

    def size(query, *args):
        nb = ctypes.c_size_t()
        assert getattr(q.load(), query)(*args, ctypes.byref(nb)) == 0
        return nb.value

    x, D, c = normal(4, 64, 28, 28), normal(16, 16, 4), codes(64, 9, 16)
    xf, Df, cf = normal(64, 1024), normal(256, 16, 4), codes(256, 300)
    W, init = normal(300, 64), normal(16, 16, 4)
    net = q.Net([q.ConvLayer(D, c, None, 64, 3, 3, 1, 1), q.PoolLayer(2, 2),
                 q.FCLayer(normal(16 * 14 * 14, 16, 4), codes(16 * 14 * 14, 40), None)], (64, 28, 28))
    return {
        "conv": (lambda **k: q.conv_forward(x, D, c, 3, 3, 1, 1, **k),
                 size("qcnn_conv_workspace_size", 4, 64, 28, 28, 64, 3, 3, 1, 1, 4, 16, 0, 0, 0)),
        "fc": (lambda **k: q.fc_forward(xf, Df, cf, **k),
               size("qcnn_fc_workspace_size", 64, 1024, 300, 4, 16, 0)),
        "net": (lambda **k: net.forward(x, **k), net.workspace_bytes(4)),
        "quantizer": (lambda **k: q.pq_quantize_fc(W, 4, 16, init, 4, **k)[0],
                      size("qcnn_pq_quantize_workspace_size", 1, 300, 64, 1, 1, 4, 16)),
    }


@pytest.mark.parametrize("raw", [False, True], ids=["object", "handle"])
@pytest.mark.parametrize("name", ["conv", "fc", "net", "quantizer"])
def test_scratch_belongs_to_the_stream_of_the_call(name, raw):
    call, scratch = _calls()[name]
    assert scratch > 0
    want = call()
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    out = torch.empty_like(want) if name != "quantizer" else None
    with torch.cuda.stream(s):
        torch.cuda._sleep(20_000_000)  # some 10 ms
    kw = {"stream": s.cuda_stream if raw else s}
    if out is not None:
        kw["out"] = out
    got = call(**kw)
    fill = [torch.full((scratch,), 255, dtype=torch.uint8, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    assert torch.equal(got, want)
    for f in fill:
        assert bool((f == 255).all())


def test_scratch_under_the_current_stream_is_a_tensor_of_it():
    """The same handle as the current stream's, by either name."""
    call, _ = _calls()["conv"]
    want = call()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        got = [call(), call(stream=s), call(stream=s.cuda_stream)]
    torch.cuda.synchronize()
    for y in got:
        assert torch.equal(y, want)
