"""Results that a call makes for another stream than the current one: memory that
the current stream has still to write is not given to them, and the copies that
error correction works on are there before its kernels."""
import pytest
import torch

import paper_1512_06473_gb300 as q

pytestmark = pytest.mark.gpu


def _late_write(nbytes):
    """A block of the current stream that is free, but written some 10 ms from now."""
    t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    torch.cuda._sleep(20_000_000)
    t.fill_(255)


@pytest.mark.parametrize("raw", [False, True], ids=["object", "handle"])
@pytest.mark.parametrize("op", ["conv", "fc", "pool", "lut", "pack", "net"])
def test_outputs_are_not_memory_of_queued_work(op, raw):
    g = torch.Generator(device="cuda").manual_seed(4)
    x = torch.randn((8, 16, 32, 32), generator=g, device="cuda")
    D = torch.randn((4, 16, 4), generator=g, device="cuda")
    c = torch.randint(0, 16, (64, 9, 4), generator=g, device="cuda", dtype=torch.uint8)
    xf = torch.randn((512, 64), generator=g, device="cuda")
    Df = torch.randn((16, 16, 4), generator=g, device="cuda")
    cf = torch.randint(0, 16, (16, 2048), generator=g, device="cuda", dtype=torch.uint8)
    net = q.Net([q.ConvLayer(D, c, None, 64, 3, 3, 1, 1), q.PoolLayer(2, 2)], (16, 32, 32))
    call = {"conv": lambda **k: q.conv_forward(x, D, c, 3, 3, 1, 1, **k),
            "fc": lambda **k: q.fc_forward(xf, Df, cf, **k),
            "pool": lambda **k: q.maxpool(x, 2, 1, **k),
            "lut": lambda **k: q.lut_build(xf, Df, **k),
            "pack": lambda **k: q.conv_pack_codes(c, 16, 3, 3, **k),
            "net": lambda **k: net.forward(x, **k)}[op]
    want = call()
    keep = want.clone()
    torch.cuda.synchronize()
    nbytes = want.untyped_storage().nbytes()
    del want
    torch.cuda.empty_cache()
    s = torch.cuda.Stream()
    _late_write(nbytes)
    got = call(stream=s.cuda_stream if raw else s)
    torch.cuda.synchronize()
    assert torch.equal(got, keep)


@pytest.mark.parametrize("kind", ["fc", "conv"])
def test_error_correction_starts_from_its_inputs(kind):
    g = torch.Generator(device="cuda").manual_seed(5)
    D = torch.randn((4, 8, 4), generator=g, device="cuda")
    if kind == "fc":
        S = torch.randn((128, 16), generator=g, device="cuda")
        T = torch.randn((128, 24), generator=g, device="cuda")
        c = torch.randint(0, 8, (4, 24), generator=g, device="cuda", dtype=torch.uint8)
        call = lambda **k: q.ec_quantize_fc(S, T, D, c, 1, 2, **k)  # noqa: E731
    else:
        S = torch.randn((4, 16, 9, 9), generator=g, device="cuda")
        T = torch.randn((4, 24, 9, 9), generator=g, device="cuda")
        c = torch.randint(0, 8, (24, 9, 4), generator=g, device="cuda", dtype=torch.uint8)
        call = lambda **k: q.ec_quantize_conv(S, T, D, c, 3, 3, 1, 1, 1, 2, **k)  # noqa: E731
    want = call()
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    torch.cuda._sleep(20_000_000)  # (the current stream is late)
    got = call(stream=s)
    s.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
