"""Every bf16 tile variant of the fused conv kernel, the 64-channel ones too, at
the edges of its channel tile (32, 64, 128), of the pairs of sub-codewords that
its table build takes together (32, 64), of odd and even runs of positions.
Integer inputs up to 4 make every table entry exact in bf16 and every sum exact,
so the result equals the reference bit for bit."""
import pytest
import torch
import torch.nn.functional as F

import paper_1512_06473_gb300 as q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c", [  # N, Cs, H, W, Ct, k, pad, C, K
    (2, 8, 9, 11, 33, 3, 1, 4, 20), (1, 12, 20, 17, 64, 3, 1, 3, 65), (3, 16, 7, 7, 65, 5, 2, 8, 33),
    (1, 4, 30, 31, 1, 2, 0, 4, 1), (2, 14, 13, 13, 129, 3, 1, 7, 128), (2, 8, 57, 3, 50, 3, 1, 4, 256),
], ids=lambda c: "x".join(map(str, c)))
def test_all_variants(c):
    N, Cs, H, W, Ct, k, pad, C, K = c
    M = Cs // C
    g = torch.Generator().manual_seed(sum(c))
    x = torch.randint(-4, 5, (N, Cs, H, W), generator=g).float()
    D = torch.randint(-4, 5, (M, K, C), generator=g).float()
    codes = torch.randint(0, K, (Ct, k * k, M), generator=g).to(torch.uint8)
    w = D[torch.arange(M), codes.long()].permute(0, 2, 3, 1).reshape(Ct, Cs, k, k)
    ref = F.conv2d(x.double(), w.double(), padding=pad)
    ran = 0
    for v, info in enumerate(q.fused_variants()):
        if not info["BF"]:
            continue
        try:
            y = q.conv_forward(x.cuda(), D.cuda(), codes.cuda(), k, k, 1, pad, algo=v, lut="bf16")
        except q.QcnnError as e:
            assert e.status == q._lib.ERR_UNSUPPORTED  # (the tile does not fit the layer)
            continue
        assert torch.equal(y.double().cpu(), ref), info
        ran += 1
    assert ran
