"""A workspace that the contraction cannot use (absent, however many bytes are
claimed, or off its alignment), for calls whose table plan needs none: the tables
run, as in a call without any."""
import pytest
import torch

import paper_1512_06473_gb300 as q

pytestmark = pytest.mark.gpu

BYTES = 64 << 20


def _fc():
    g = torch.Generator(device="cuda").manual_seed(21)
    N, Cs, Ct, C, K = 256, 64, 4096, 4, 32
    x = torch.randn((N, Cs), generator=g, device="cuda")
    D = torch.randn((Cs // C, K, C), generator=g, device="cuda")
    c = torch.randint(0, K, (Cs // C, Ct), generator=g, device="cuda", dtype=torch.uint8)
    y = torch.empty((N, Ct), device="cuda")
    bits = q.fc_pack_codes(c, K)

    def call(codes, fn):
        return lambda ws, n: fn(x.data_ptr(), N, Cs, Ct, D.data_ptr(), C, K, codes.data_ptr(), None,
                                y.data_ptr(), 0, 0, ws, n, torch.cuda.current_stream().cuda_stream)
    return y, call(c, q.load().qcnn_fc_forward), call(bits, q.load().qcnn_fc_forward_packed), x, D, c


def _conv():
    g = torch.Generator(device="cuda").manual_seed(22)
    N, Cs, H, Ct, C, K = 2, 64, 56, 64, 4, 128
    x = torch.randn((N, Cs, H, H), generator=g, device="cuda")
    D = torch.randn((Cs // C, K, C), generator=g, device="cuda")
    c = torch.randint(0, K, (Ct, 9, Cs // C), generator=g, device="cuda", dtype=torch.uint8)
    return x, D, q.conv_pack_codes(c, K, 3, 3), Ct


def _unusable():
    buf = torch.empty(BYTES + 256, dtype=torch.uint8, device="cuda")
    return {"absent": (None, BYTES), "misaligned": (buf.data_ptr() + 8, BYTES), "none": (None, 0)}, buf


def test_fc():
    y, byte_codes, bit_codes, *keep = _fc()
    ways, buf = _unusable()
    for fn in (byte_codes, bit_codes):
        got = {}
        for name, (ws, n) in ways.items():
            assert fn(ws, n) == 0, name
            got[name] = y.clone()
        assert torch.equal(got["absent"], got["none"])
        assert torch.equal(got["misaligned"], got["none"])


def test_conv_and_net():
    x, D, packed, Ct = _conv()
    table = q.conv_plan(2, 64, 56, 56, 64, 3, 3, 1, 1, 4, 128)
    want = q.conv_forward(x, D, packed, 3, 3, 1, 1, packed=True, Ct=Ct, algo=table["algo"])
    y = torch.empty_like(want)
    net = q.Net([q.ConvLayer(D, packed, None, Ct, 3, 3, 1, 1, relu=False, packed=True)], (64, 56, 56))
    lib, st = q.load(), torch.cuda.current_stream().cuda_stream
    ways, buf = _unusable()
    for name, (ws, n) in ways.items():
        y.zero_()
        assert lib.qcnn_conv_forward(x.data_ptr(), 2, 64, 56, 56, Ct, 3, 3, 1, 1, D.data_ptr(), 4, 128,
                                     packed.data_ptr(), 1, None, y.data_ptr(), 0, 0, 0, ws, n, st) == 0
        assert torch.equal(y, want), name
        y.zero_()
        assert lib.qcnn_net_forward(net._arr, 1, x.data_ptr(), 2, 64, 56, 56, y.data_ptr(), ws, n,
                                    st) == 0, name
        assert torch.equal(y, want), name
