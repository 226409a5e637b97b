"""What AUTO runs, by the host-side route queries: the contraction's plans within
their bounds over random shapes, and the route queries against the plan queries."""
import ctypes
import random

import pytest

import bench  # noqa: E402
import paper_1512_06473_gb300 as q
import synth
from paper_1512_06473_gb300 import _lib


def scratch(algo, args):
    nb = ctypes.c_size_t()
    st = q.load().qcnn_conv_workspace_size(*args, _lib.CODES_PACKED, _lib.ALGO[algo], 0,
                                           ctypes.byref(nb))
    return nb.value if st == _lib.OK else None


def test_contract_plans_are_within_their_bounds():
    """Tiles of 16 .. 192 columns in steps of 16, at most 64 splits, a grid of at most
    one CTA per SM; scratch for the pieces of inputs (6 bytes a component, padded to
    16 terms) and codebooks, 2 GB and the splits' partial sums at most."""
    r = random.Random(3)
    took = 0
    for _ in range(300):
        C, k, s = r.randint(1, 8), r.choice([1, 2, 3, 5, 7, 11]), r.choice([1, 1, 2, 4])
        M, pad, K = r.randint(1, 64), r.choice([0, k // 2]), r.choice([1, 16, 100, 256])
        N, H, W, Ct = r.randint(1, 128), r.randint(k, 120), r.randint(k, 120), r.randint(1, 600)
        args = (N, M * C, H, W, Ct, k, k, s, pad, C, K)
        if N * M * C * H * W > 2 ** 30:
            continue
        need = scratch("contract", args)
        if need is None:
            continue
        p = q.conv_route(*args[:9], Csp=C, K=K, algo="contract")
        assert p["algo"] == "contract" and p["variant"] == -1 and p["cluster"] == 1, args
        assert p["positions"] % 16 == 0 and 16 <= p["positions"] <= 192, args
        assert 1 <= p["splits"] <= 64 and 1 <= p["ctas"] <= 152 and p["channels"] == 128, args
        Ho, Wo = (H + 2 * pad - k) // s + 1, (W + 2 * pad - k) // s + 1
        parts = 4 * p["splits"] * N * Ct * Ho * Wo if p["splits"] > 1 else 0
        least = (0 if k < s else 6 * N * M * C * Ho * Wo) + parts
        assert least <= need <= (2 << 30) + parts + 64 * 300 * 257 * 1024, args
        took += 1
    assert took >= 100


def test_more_than_16_stride_phases_are_not_contracted():
    args = (2, 16, 40, 40, 32, 5, 5, 5, 0, 4, 16)
    assert scratch("contract", args) is None
    assert q.conv_route(*args[:9], Csp=4, K=16)["algo"] != "contract"


def test_routes_of_the_benchmark():
    """Batch 128 of the AlexNet-shaped stack is contracted throughout; FC layers of
    one image, and tables of bfloat16 entries, are not."""
    w = synth.alexnet()
    assert bench.layer_routes(q, w, 128) == ["contract", None, "contract", None, "contract",
                                             "contract", "contract", None, "contract", "contract",
                                             "contract"]
    assert bench.layer_routes(q, w, 1)[-3:] == ["tables"] * 3
    assert q.conv_route(8, 64, 56, 56, 64, 3, 3, 1, 1, lut="bf16")["algo"] == "fused"
    assert q.fc_route(128, 4096, 1000, lut="bf16")["algo"] == "tables"


def test_a_route_that_is_not_the_contraction_is_the_plan():
    for args in [(1, 64, 28, 28, 64, 3, 3, 1, 1), (1, 64, 56, 56, 64, 3, 3, 2, 1)]:
        for lut in ("fp32", "bf16"):
            assert q.conv_route(*args, lut=lut) == q.conv_plan(*args, lut=lut), (args, lut)
    for algo in ("fused", "unfused", "chunked", "phase", "contract"):
        args = (8, 64, 28, 28, 64, 3, 3, 1, 1)
        assert q.conv_route(*args, algo=algo) == q.conv_plan(*args, algo=algo)
    t, p = q.fc_route(1, 4096, 4096), q.fc_plan(1, 4096, 4096)
    assert {k: t[k] for k in ("images", "outputs", "splits", "ctas", "cluster")} == \
        {k: p[k] for k in ("images", "outputs", "splits", "ctas", "cluster")}


def test_errors():
    lib = q.load()
    i6, i8 = (ctypes.c_int * 6)(), (ctypes.c_int * 8)()
    assert lib.qcnn_fc_route_info(2, 12, 4, 3, 16, 0, None) == _lib.ERR_INVALID_ARG
    assert lib.qcnn_fc_route_info(2, 10, 4, 3, 16, 0, i6) == _lib.ERR_INVALID_ARG
    args = (2, 8, 9, 9, 4, 3, 3, 2, 1, 4, 16, 1)
    assert lib.qcnn_conv_route_info(*args, 0, 0, None) == _lib.ERR_INVALID_ARG
    assert lib.qcnn_conv_route_info(*args, 1, 0, i8) == _lib.ERR_UNSUPPORTED  # fused, stride 2
    assert lib.qcnn_conv_route_info(*args, 0, 0, i8) == _lib.OK


def test_contracted_stages_are_against_the_tensor_roof():
    """Six bf16 products per multiply-add: conv2 at batch 128 in exactly that time."""
    from paper_1512_06473_gb300 import costmodel as cm
    w = synth.alexnet()
    L, (sin, sout) = w.layers[2], w.shapes()[2]
    c = cm.conv_cost(L.Cs, L.Ct, sin[1], sin[2], L.kh, L.kw, sout[1], sout[2], L.Csp, L.K)
    ms = 12.0 * 128 * c.dense_macs / 1900e12 * 1e3
    st = bench.stage_rooflines(w, cm, [ms] * len(w.layers), 128, 40000.0, 6700.0,
                               bench.layer_routes(q, w, 128), 1900.0)
    assert st[2]["bound"] == "tensor" and st[2]["frac"] == pytest.approx(1.0, rel=1e-3)
    assert st[1]["bound"] == "hbm"


def test_both_sides_of_the_dispatch():
    """Short calls keep their tables; their larger neighbours do not."""
    def conv(*a):
        return q.conv_route(*a[:9], Csp=a[9], K=a[10])["algo"]
    assert conv(1, 64, 56, 56, 64, 3, 3, 1, 1, 4, 128) == "fused"
    assert conv(1, 64, 56, 56, 128, 3, 3, 1, 1, 4, 128) == "contract"
    assert conv(1, 64, 56, 56, 64, 3, 3, 2, 1, 4, 128) == "phase"
    assert conv(1, 3, 227, 227, 96, 11, 11, 4, 0, 3, 128) == "contract"
    assert conv(1, 64, 28, 28, 64, 1, 1, 1, 0, 4, 128) == "fused"
    assert conv(1, 128, 56, 56, 64, 1, 1, 1, 0, 4, 128) == "contract"
    assert conv(2, 44, 30, 30, 476, 1, 1, 1, 0, 4, 32) == "contract"
    assert conv(4, 20, 14, 14, 259, 1, 1, 2, 0, 4, 32) == "contract"
    assert q.fc_route(32, 1024, 1024)["algo"] == "tables"
    assert q.fc_route(64, 512, 256, K=16)["algo"] == "tables"
    assert q.fc_route(64, 1024, 300)["algo"] == "contract"
    assert q.fc_route(64, 4096, 1000)["algo"] == "contract"
    assert q.fc_route(24, 4096, 4096)["algo"] == "tables"
    assert q.fc_route(9, 4096, 4096, K=64)["algo"] == "contract"
