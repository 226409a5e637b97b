"""Sums that are not finite, taken again by plain arithmetic after the contraction:
every place of a tile (both halves of its columns, ragged ends), split sub-spaces,
strides, FC rows and 1x1 kernels, with ReLU, and outputs of which all are infinite."""
import pytest
import torch
import torch.nn.functional as F

import paper_1512_06473_gb300 as q

pytestmark = pytest.mark.gpu

INF = float("inf")


def weights(D, codes, k):
    M, K, C = D.shape
    w = D.double()[torch.arange(M, device=D.device), codes.long()]
    return w.permute(0, 2, 3, 1).reshape(codes.shape[0], M * C, k, k)


def agree(y, x, w, b, relu, **kw):
    """y is non-finite where the sums of products are, by the terms that exist (a
    zero of the padding is no term), and within 1e-5 of the largest elsewhere."""
    hot = torch.where(torch.isfinite(x), 0.0, x).double()
    finite = F.conv2d(torch.where(torch.isfinite(x), x, 0.0).double(), w, b.double(), **kw)
    plus = F.conv2d((hot == INF).double(), (w > 0).double(), **kw) + \
        F.conv2d((hot == -INF).double(), (w < 0).double(), **kw)
    minus = F.conv2d((hot == INF).double(), (w < 0).double(), **kw) + \
        F.conv2d((hot == -INF).double(), (w > 0).double(), **kw)
    nan = F.conv2d(torch.isnan(x).double(), torch.ones_like(w), **kw) + \
        F.conv2d((hot.abs() == INF).double(), (w == 0).double(), **kw)
    ref = finite.clone()
    ref[plus > 0.5] = INF
    ref[minus > 0.5] = -INF
    ref[(nan > 0.5) | ((plus > 0.5) & (minus > 0.5))] = float("nan")
    if relu:
        ref = torch.where(torch.isnan(ref), 0.0, ref.clamp(min=0))  # (as the tables: max(NaN, 0))
    y = y.double().reshape(ref.shape)
    ok = torch.isfinite(ref)
    assert torch.equal(torch.isnan(y), torch.isnan(ref))
    assert torch.equal(y[torch.isinf(ref)], ref[torch.isinf(ref)])
    assert bool(((y - ref)[ok].abs() <= 1e-5 * finite.abs().max()).all())
    return int((~ok).sum())


def data(N, Cs, H, W, Ct, k, C, K, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((N, Cs, H, W), generator=g, device="cuda")
    D = torch.randn((Cs // C, K, C), generator=g, device="cuda")
    D[0, 0, 0] = 0.0
    c = torch.randint(0, K, (Ct, k * k, Cs // C), generator=g, device="cuda", dtype=torch.uint8)
    b = torch.randn((Ct,), generator=g, device="cuda")
    at = torch.rand(x.shape, generator=g, device="cuda")
    return x, D, c, b, at


@pytest.mark.parametrize("relu", [False, True])
@pytest.mark.parametrize("share", [0.002, 1.0])
@pytest.mark.parametrize("case", [  # N, Cs, H, W, Ct, k, stride, pad, C, K
    (2, 12, 13, 11, 150, 3, 1, 1, 4, 16),
    (1, 200, 9, 9, 40, 3, 1, 1, 8, 33),     # split sub-spaces
    (1, 3, 39, 31, 24, 11, 4, 0, 3, 32),    # stride phases that share blocks
    (2, 16, 21, 19, 33, 3, 2, 1, 8, 16),
    (3, 20, 17, 15, 130, 1, 1, 0, 4, 16),   # one-step blocks
], ids=lambda c: "x".join(map(str, c)))
def test_conv(case, share, relu):
    N, Cs, H, W, Ct, k, s, p, C, K = case
    x, D, c, b, at = data(N, Cs, H, W, Ct, k, C, K, sum(case))
    x[at < share / 3] = INF
    x[(at >= share / 3) & (at < 2 * share / 3)] = -INF
    x[(at >= 2 * share / 3) & (at < share)] = float("nan")
    y = q.conv_forward(x, D, c, k, k, s, p, b, relu=relu, algo="contract")
    agree(y, x, weights(D, c, k), b, relu, stride=s, padding=p)
    x = torch.randn_like(x)
    x[at < share] = INF  # (no cancellation: infinite sums, not NaN)
    D, w = D.abs() + 0.5, None
    y = q.conv_forward(x, D, c, k, k, s, p, b, relu=relu, algo="contract")
    bad = agree(y, x, weights(D, c, k), b, relu, stride=s, padding=p)
    assert bad == y.numel() if share == 1.0 else bad > 0


def test_a_codebook_with_an_infinity():
    x, D, c, b, _ = data(2, 16, 9, 9, 140, 3, 4, 16, 3)
    D[1, 5, 2] = INF
    x = x.abs() + 0.5
    y = q.conv_forward(x, D, c, 3, 3, 1, 1, b, algo="contract")
    r = q.conv_forward(x, D, c, 3, 3, 1, 1, b, algo="unfused")
    assert torch.equal(torch.isinf(y), torch.isinf(r)) and not bool(torch.isnan(y).any())
    assert 0 < int(torch.isinf(y).sum()) < y.numel()


def test_every_output_of_a_large_layer():
    """All sums infinite, several tiles to a CTA: no wait of the kernel's other warps
    runs out meanwhile."""
    N, M, Ct, C, K = 256, 16384, 4096, 4, 16
    g = torch.Generator(device="cuda").manual_seed(9)
    x = torch.randn((N, M * C), generator=g, device="cuda")
    x[:, 3] = INF
    D = torch.randn((M, K, C), generator=g, device="cuda")
    c = torch.randint(0, K, (M, Ct), generator=g, device="cuda", dtype=torch.uint8)
    q.device_check()
    y = q.fc_forward(x, D, c)
    assert q.device_check() == 0
    sign = torch.sign(D[0][c[0].long()][:, 3])
    assert bool((sign != 0).all())
    assert torch.equal(y, (sign * INF).expand(N, Ct))
