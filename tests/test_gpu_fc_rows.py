"""FC byte codes whose rows begin at every offset from a 16-byte boundary (Ct mod
16), on the contraction's side of the dispatch, and whole arrays off it (the
tables).  Integer inputs up to 8: every sum is exact."""
import pytest
import torch

import paper_1512_06473_gb300 as q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ct", list(range(1, 18)) + [111, 113, 127, 130, 249, 251, 263, 385, 1001])
@pytest.mark.parametrize("N,C,M", [(200, 4, 37), (320, 8, 21), (1000, 3, 8)])
def test_rows(Ct, N, C, M):
    K = 256
    g = torch.Generator(device="cuda").manual_seed(Ct * 10 + C)
    x = torch.randint(-8, 9, (N, M * C), generator=g, device="cuda").float()
    D = torch.randint(-8, 9, (M, K, C), generator=g, device="cuda").float()
    c = torch.randint(0, K, (M, Ct), generator=g, device="cuda", dtype=torch.uint8)
    w = D.double()[torch.arange(M, device="cuda")[:, None], c.long()]  # [M, Ct, C]
    want = torch.einsum("nmj,mcj->nc", x.double().view(N, M, C), w)
    assert torch.equal(q.fc_forward(x, D, c).double(), want)
    off = torch.empty(c.numel() + 3, dtype=torch.uint8, device="cuda")[3:].view(M, Ct).copy_(c)
    assert torch.equal(q.fc_forward(x, D, off).double(), want)
