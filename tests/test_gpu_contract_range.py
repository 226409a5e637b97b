"""The contraction over fp32's exponent range: inputs and codebooks near its lower
end (subnormal ones too) and so large that the sums go to plain arithmetic.

Bound: as for values of order one, (14 + G / 2) 2^-23 S with S = sum |d||x| + |b|
and G groups (12 accumulations of at most 2^-23 each in a group, products left out
below 3 * 2^-25, groups added with 2^-24 each); plus 2^-150 for each rounding to a
subnormal, of which there is one per partial sum (64 at most) and one at the end.
Plain arithmetic (the largest scales) adds n terms in fp32: n 2^-24 S."""
import pytest
import torch
import torch.nn.functional as F

import paper_1512_06473_gb300 as q

pytestmark = pytest.mark.gpu

# exponents of inputs and codebooks
SCALES = [(-112, 0), (-120, 0), (-126, 0), (-132, 0), (-140, 3), (0, -112), (0, -120), (2, -130),
          (-70, -70), (-126, 70), (70, -126), (-60, -84), (60, 30), (114, 0), (20, 90), (-20, 120)]


@pytest.mark.parametrize("case", [  # N, Cs, H, Ct, k, C, K
    (2, 24, 11, 40, 3, 4, 32), (1, 160, 6, 20, 3, 8, 16), (40, 60, 1, 130, 1, 3, 16)],
    ids=lambda c: "x".join(map(str, c)))
@pytest.mark.parametrize("ex,ed", SCALES)
def test_scales(ex, ed, case):
    N, Cs, H, Ct, k, C, K = case
    g = torch.Generator().manual_seed(ex * 31 + ed + Cs)
    M = Cs // C
    x = torch.ldexp(torch.randn((N, Cs, H, H), generator=g).double(), torch.tensor(ex)).float()
    D = torch.ldexp(torch.randn((M, K, C), generator=g).double(), torch.tensor(ed)).float()
    codes = torch.randint(0, K, (Ct, k * k, M), generator=g).to(torch.uint8)
    b = torch.zeros(Ct)
    w = D.double()[torch.arange(M), codes.long()].permute(0, 2, 3, 1).reshape(Ct, Cs, k, k)
    ref = F.conv2d(x.double(), w, padding=k // 2)
    S = F.conv2d(x.double().abs(), w.abs(), padding=k // 2)
    assert float(S.max()) < 2.0 ** 127
    y = q.conv_forward(x.cuda(), D.cuda(), codes.cuda(), k, k, 1, k // 2, b.cuda(), algo="contract")
    n = Cs * k * k
    bound = max(14 + n / 32, n / 2) * 2.0 ** -23 if max(ex, ed, ex + ed) > 80 else \
        (14 + n / 32) * 2.0 ** -23
    assert bool(((y.double().cpu() - ref).abs() <= bound * S + 65 * 2.0 ** -150).all())
