"""The tensor-core contraction (algo "contract", and the FC and AUTO calls that
take it) where its tiling can go wrong: edges of the channel tile (128), of the
column tile (16 .. 192), of blocks of 16 terms, of groups of two steps, of the
clusters' shared copies; every C's; strides whose phases fill blocks or share
them; sub-space ranges that are split.

Integer inputs up to 8 make every product and partial sum exact, so the result
equals the reference bit for bit.  For others the bound is worked out from the
arithmetic: an operand's three bf16 pieces are exact and the products left out
are below 3 * 2^-25 of |x||d|; a group of 32 terms is 12 accumulations with at
most 2^-23 of the group's magnitude lost in each; groups (and splits) are added
with 2^-24 of the running magnitude each.  With S = sum |d||x| + |b| and G
groups that is less than (14 + G / 2) 2^-23 S per output."""
import ctypes

import pytest
import torch
import torch.nn.functional as F

import paper_1512_06473_gb300 as q

pytestmark = pytest.mark.gpu


def draw(shape, integer, gen, scale=1.0):
    if integer:
        return torch.randint(-8, 9, shape, generator=gen).float()
    return torch.randn(shape, generator=gen) * scale


def case(Cs, Ct, kk, C, K, xshape, integer, seed):
    gen = torch.Generator().manual_seed(seed)
    M = Cs // C
    x = draw(xshape, integer, gen)
    D = draw((M, K, C), integer, gen, 0.5)
    b = draw((Ct,), integer, gen, 0.1)
    codes = torch.randint(0, K, (Ct, kk, M), generator=gen).to(torch.uint8)
    return x, D, b, codes


def weights(D, codes, kh, kw):
    M, K, C = D.shape
    w = D.double()[torch.arange(M), codes.long()]  # [Ct, kk, M, C]
    return w.permute(0, 2, 3, 1).reshape(codes.shape[0], M * C, kh, kw)


def check(y, x, w, b, relu, integer, **kw):
    x, b = x.double(), b.double()
    ref = F.conv2d(x, w, b, **kw)
    S = F.conv2d(x.abs(), w.abs(), b.abs(), **kw)
    groups = w[0].numel() / 16  # of one step: more than there are
    if relu:
        ref = ref.relu()
    y = y.double().cpu().reshape(ref.shape)
    if integer:
        assert torch.equal(y, ref)
    else:
        assert bool(((y - ref).abs() <= (14 + groups / 2) * 2.0 ** -23 * S).all())


# N, Cs, H, W, Ct, kh, kw, stride, pad, C, K
CONV = [
    (1, 1, 1, 1, 1, 1, 1, 1, 0, 1, 1),          # one term, one output
    (1, 4, 5, 5, 3, 3, 3, 1, 1, 4, 5),
    (2, 12, 13, 13, 127, 3, 3, 1, 1, 4, 128),   # a block short of a sub-vector
    (1, 20, 9, 9, 129, 3, 3, 1, 1, 4, 256),     # one channel past the tile
    (3, 16, 7, 9, 128, 2, 4, 1, 0, 8, 33),      # two quarters a sub-vector
    (2, 30, 8, 8, 130, 3, 3, 1, 1, 5, 64),      # C's 5: zeros between
    (2, 14, 8, 11, 65, 3, 3, 1, 2, 7, 20),
    (1, 9, 12, 12, 40, 3, 3, 1, 1, 3, 16),
    (2, 10, 6, 6, 33, 3, 3, 1, 1, 2, 2),
    (5, 8, 7, 7, 257, 1, 1, 1, 0, 4, 32),       # one tap, stages of two blocks
    (1, 72, 15, 13, 48, 1, 1, 1, 0, 8, 16),     # the last stage of one block
    (2, 16, 31, 29, 96, 3, 3, 2, 1, 8, 64),     # phases of 4, 2, 2, 1 taps
    (1, 3, 39, 39, 24, 11, 11, 4, 0, 3, 128),   # 16 phases of one sub-vector share blocks
    (2, 6, 23, 19, 20, 5, 5, 3, 2, 6, 64),
    (1, 8, 9, 9, 16, 1, 1, 2, 0, 4, 16),        # one tap of one phase
    (1, 4, 17, 17, 16, 3, 3, 5, 1, 4, 16),      # stride past the kernel
    (1, 8, 6, 7, 12, 1, 1, 1, 1, 4, 16),        # padding past the kernel
    (2, 128, 13, 13, 200, 3, 3, 1, 1, 8, 128),  # split into ranges of sub-spaces
    (40, 4, 6, 6, 16, 3, 3, 1, 1, 4, 16),       # tiles across many images
]


@pytest.mark.parametrize("integer", [True, False], ids=["integer", "normal"])
@pytest.mark.parametrize("c", CONV, ids=lambda c: "x".join(map(str, c)))
def test_conv(c, integer):
    N, Cs, H, W, Ct, kh, kw, s, p, C, K = c
    x, D, b, codes = case(Cs, Ct, kh * kw, C, K, (N, Cs, H, W), integer, sum(c))
    w = weights(D, codes, kh, kw)
    dx, dD, db, dc = x.cuda(), D.cuda(), b.cuda(), codes.cuda()
    for packed in (False, True):
        cc = q.conv_pack_codes(dc, K, kh, kw) if packed else dc
        y = q.conv_forward(dx, dD, cc, kh, kw, s, p, db, relu=packed, algo="contract",
                           packed=packed, Ct=Ct)
        check(y, x, w, b, packed, integer, stride=s, padding=p)
    # inputs and codes off the wide loads' alignment
    xo = torch.empty(x.numel() + 1, device="cuda")[1:].view(x.shape).copy_(x)
    co = torch.empty(codes.numel() + 3, dtype=torch.uint8, device="cuda")[3:].view(codes.shape)
    co.copy_(codes)
    Do = torch.empty(D.numel() + 1, device="cuda")[1:].view(D.shape).copy_(D)
    y = q.conv_forward(xo, Do, co, kh, kw, s, p, db, algo="contract")
    check(y, x, w, b, False, integer, stride=s, padding=p)


# N, Cs, Ct, C, K: all on the contraction's side of the dispatch
FC = [
    (32, 4, 1, 4, 3),         # one block, one channel
    (33, 60, 128, 4, 16),     # the last block a sub-vector short
    (9, 256, 129, 4, 64),     # two tiles share copies; the second of one channel
    (47, 272, 385, 8, 200),   # four; the last stage of one block
    (64, 600, 301, 3, 16),    # codes copied byte by byte
    (193, 104, 520, 8, 256),  # past the widest column tile; a tile is absent
    (70, 2304, 513, 4, 5),    # many stages: each buffer used again and again
    (40, 1001, 130, 7, 33),
    (64, 640, 300, 1, 2),
]


@pytest.mark.parametrize("integer", [True, False], ids=["integer", "normal"])
@pytest.mark.parametrize("c", FC, ids=lambda c: "x".join(map(str, c)))
def test_fc(c, integer):
    N, Cs, Ct, C, K = c
    x, D, b, codes = case(Cs, Ct, 1, C, K, (N, Cs, 1, 1), integer, sum(c))
    w = weights(D, codes, 1, 1)
    codes = codes[:, 0].t().contiguous().cuda()  # [M, Ct]
    xf = x.view(N, Cs).cuda()
    got = [q.fc_forward(xf, D.cuda(), cc, b.cuda(), relu=True, Ct=Ct)
           for cc in (codes, q.fc_pack_codes(codes, K))]
    check(got[0], x, w, b, True, integer)
    assert torch.equal(got[0], got[1])


@pytest.mark.parametrize("N,H,Ct", [(2, 9, 40), (32, 40, 130)])
def test_non_finite_inputs_stay_where_the_lookups_put_them(N, H, Ct):
    """Zero-weight padding terms must not spread an infinity: the outputs that
    are NaN or infinite are those of the table path."""
    Cs, W, C, K = 12, H, 4, 16
    x, D, b, codes = case(Cs, Ct, 9, C, K, (N, Cs, H, W), False, 5)
    x[0, 3, 4, 4], x[N - 1, 7, 0, 8], x[1, 0, 8, 0] = float("inf"), float("-inf"), float("nan")
    D[2, 3], D[1, 5, 1] = 2.0, 0.0
    args = (x.cuda(), D.cuda(), codes.cuda(), 3, 3, 1, 1, b.cuda())
    y = q.conv_forward(*args, algo="contract")
    r = q.conv_forward(*args, algo="unfused")
    fin = torch.isfinite(r)
    assert 0 < int((~fin).sum()) < fin.numel() // 2
    assert torch.equal(torch.isnan(y), torch.isnan(r))
    assert torch.equal(y[torch.isinf(r)], r[torch.isinf(r)])
    assert bool(((y - r)[fin].abs() <= 1e-5 * r[fin].abs().max()).all())


def test_workspace_of_the_tables_plan_is_still_enough():
    """AUTO with the scratch that its table plan needs runs that plan, bit for
    bit; with less it is refused."""
    N, Cs, H, W, Ct, C, K = 8, 64, 28, 28, 64, 4, 256
    x, D, b, codes = case(Cs, Ct, 9, C, K, (N, Cs, H, W), False, 6)
    args = (x.cuda(), D.cuda(), codes.cuda(), 3, 3, 1, 1, b.cuda())
    plan = q.conv_plan(N, Cs, H, W, Ct, 3, 3, 1, 1, C, K, packed=False)
    ref = q.conv_forward(*args, algo=plan["algo"])
    need = {}
    for algo in ("auto", plan["algo"]):
        nb = ctypes.c_size_t()
        assert q.load().qcnn_conv_workspace_size(N, Cs, H, W, Ct, 3, 3, 1, 1, C, K, 0,
                                                 q._lib.ALGO[algo], 0, ctypes.byref(nb)) == 0
        need[algo] = nb.value
    tables = need[plan["algo"]]
    assert 256 < tables < need["auto"]
    ws = torch.empty(tables, dtype=torch.uint8, device="cuda")
    assert torch.equal(q.conv_forward(*args, workspace=ws), ref)
    with pytest.raises(q.QcnnError):
        q.conv_forward(*args, workspace=ws[:256])


def test_captured_calls_read_their_inputs_at_replay():
    x, D, b, codes = case(64, 200, 9, 4, 64, (3, 64, 13, 13), True, 7)
    xd, ws = x.cuda(), torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    args = (xd, D.cuda(), codes.cuda(), 3, 3, 1, 1, b.cuda())
    q.conv_forward(*args, algo="contract", workspace=ws)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        y = q.conv_forward(*args, algo="contract", workspace=ws)
    for seed in (8, 9):
        x = draw(x.shape, True, torch.Generator().manual_seed(seed))
        xd.copy_(x)
        g.replay()
        torch.cuda.synchronize()
        check(y, x, weights(D, codes, 3, 3), b, False, True, padding=1)


def test_fc_workspace_of_the_tables_plan_is_still_enough():
    """As above for an FC layer; the tables' result comes from the call that
    never contracts (the same plan: its partial sums fit its scratch)."""
    N, Cs, Ct, C, K = 64, 1024, 300, 4, 32
    x, D, b, codes = case(Cs, Ct, 1, C, K, (N, Cs, 1, 1), False, 10)
    x, D, b = x.view(N, Cs).cuda(), D.cuda(), b.cuda()
    codes = codes[:, 0].t().contiguous().cuda()
    plan = q.fc_plan(N, Cs, Ct, C, K)
    groups = plan["splits"] // plan["cluster"]
    tables = groups * N * Ct * 4 if groups > 1 else 0
    nb = ctypes.c_size_t()
    assert q.load().qcnn_fc_workspace_size(N, Cs, Ct, C, K, 0, ctypes.byref(nb)) == 0
    assert 256 < tables < nb.value
    ref = torch.empty((N, Ct), device="cuda")
    assert q.load().qcnn_fc_forward_noalloc(x.data_ptr(), N, Cs, Ct, D.data_ptr(), C, K,
                                            codes.data_ptr(), b.data_ptr(), ref.data_ptr(), 0,
                                            torch.cuda.current_stream().cuda_stream) == 0
    ws = torch.empty(tables, dtype=torch.uint8, device="cuda")
    assert torch.equal(q.fc_forward(x, D, codes, b, workspace=ws), ref)
    with pytest.raises(q.QcnnError):
        q.fc_forward(x, D, codes, b, workspace=ws[:256])
