"""FC layers on the contraction's side of the dispatch, where its tiling can go wrong:
edges of the channel tile (128) and of the column tile (16 .. 192), a last block
short of a sub-vector, a last stage of one block, many stages; byte and bit-packed
codes.  Integer inputs up to 8 give exact sums; for others the bound of the
contraction's arithmetic, (14 + G / 2) 2^-23 S with S = sum |d||x| + |b| and G groups."""
import pytest
import torch

import paper_1512_06473_gb300 as q

pytestmark = pytest.mark.gpu

# N, Cs, Ct, C, K
FC = [
    (2048, 16, 1, 4, 256),    # two stages, one channel
    (513, 60, 128, 4, 256),   # the last block a sub-vector short
    (400, 256, 129, 4, 64),   # a second channel tile of one channel
    (47, 1072, 385, 8, 200),  # the last stage of one block
    (300, 600, 301, 3, 64),   # C's 3, rows at every offset
    (193, 208, 520, 8, 256),  # a last column tile of one image
    (70, 9216, 513, 4, 16),   # many stages: each buffer used again and again
    (40, 1001, 130, 7, 250),
    (1000, 128, 300, 1, 7),   # C's 1, three-bit codes
]


@pytest.mark.parametrize("integer", [True, False], ids=["integer", "normal"])
@pytest.mark.parametrize("c", FC, ids=lambda c: "x".join(map(str, c)))
def test_fc(c, integer):
    N, Cs, Ct, C, K = c
    assert q.fc_route(N, Cs, Ct, C, K)["algo"] == "contract"
    M = Cs // C
    g = torch.Generator(device="cuda").manual_seed(sum(c))

    def values(*shape):
        if integer:
            return torch.randint(-8, 9, shape, generator=g, device="cuda").float()
        return torch.randn(shape, generator=g, device="cuda")

    x, D, b = values(N, Cs), values(M, K, C), values(Ct)
    codes = torch.randint(0, K, (M, Ct), generator=g, device="cuda", dtype=torch.uint8)
    w = D.double()[torch.arange(M, device="cuda")[:, None], codes.long()]  # [M, Ct, C]
    xd = x.double().view(N, M, C)
    want = (torch.einsum("nmj,mcj->nc", xd, w) + b.double()).relu()
    S = torch.einsum("nmj,mcj->nc", xd.abs(), w.abs()) + b.double().abs()
    y = q.fc_forward(x, D, codes, b, relu=True)
    if integer:
        assert torch.equal(y.double(), want)
    else:
        groups = M * (2 if C > 4 else 1) / 8 + 1
        assert bool(((y.double() - want).abs() <= (14 + groups / 2) * 2.0 ** -23 * S).all())
    assert torch.equal(q.fc_forward(x, D, q.fc_pack_codes(codes, K), b, relu=True, Ct=Ct), y)
