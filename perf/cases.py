"""The calls whose speed counts: single product-quantized layers, a whole
network at both ends of its batch range, and the quantizer, each through the
package's public entry points.

A case is a dict of plain values; ``op`` says which entry point runs it:
  fc      fc_forward         (byte codes, or bit-packed rows with ``bits``)
  conv    conv_forward       (codes packed at load, or canonical ones)
  net     Net.forward        (the AlexNet-shaped stack: 227x227x3 -> 1000 logits)
  kmeans  pq_quantize_conv   (dense kernels -> codebooks and codes)
Sizes are those of the AlexNet-, VGG-16-shaped and single-layer workloads of
this repository, and ragged ones between them.
"""
import math

import torch
import torch.nn.functional as F

import paper_1512_06473_gb300 as q

# AlexNet-shaped stack (ungrouped): Ct, kernel, stride, pad, C's, K, then pools
ALEX = [("conv", 96, 11, 4, 0, 3, 128), ("pool", 3, 2), ("conv", 256, 5, 1, 2, 4, 128),
        ("pool", 3, 2), ("conv", 384, 3, 1, 1, 4, 128), ("conv", 384, 3, 1, 1, 4, 128),
        ("conv", 256, 3, 1, 1, 4, 128), ("pool", 3, 2), ("fc", 4096, 4, 32, True),
        ("fc", 4096, 4, 32, True), ("fc", 1000, 4, 32, False)]
ALEX_IN = (3, 227, 227)


def _fc(name, N, Cs, Ct, Csp, K, bits=False, relu=True):
    return {"name": name, "op": "fc", "N": N, "Cs": Cs, "Ct": Ct, "Csp": Csp, "K": K,
            "bits": bits, "relu": relu}


def _conv(name, N, Cs, H, W, Ct, k, stride, pad, Csp, K, packed=True, lut="fp32", relu=True):
    return {"name": name, "op": "conv", "N": N, "Cs": Cs, "H": H, "W": W, "Ct": Ct, "k": k,
            "stride": stride, "pad": pad, "Csp": Csp, "K": K, "packed": packed, "lut": lut,
            "relu": relu}


def listed():
    return [
        # the smallest call: one classifier-sized layer for a handful of inputs
        _fc("fc512_b8", 8, 512, 256, 4, 16, relu=False),
        # the largest FC layer while serving one image: latency, and the codes' bytes
        _fc("fc6_b1", 1, 9216, 4096, 4, 32),
        # an FC layer of a served batch from codes stored in ceil(log2 K) bits
        _fc("fc7_bits_b64", 64, 4096, 4096, 4, 32, bits=True),
        # the largest FC layer at the largest batch
        _fc("fc6_b256", 256, 9216, 4096, 4, 32),
        # one 3x3 layer on one image: launches and too few blocks
        _conv("conv56_b1", 1, 64, 56, 56, 64, 3, 1, 1, 4, 128, relu=False),
        # the strided first layer of an image network, a medium batch
        _conv("conv1_s4_b32", 32, 3, 227, 227, 96, 11, 4, 0, 3, 128),
        # a VGG layer with 8-wide sub-vectors at a served batch
        _conv("vgg28_b32", 32, 256, 28, 28, 512, 3, 1, 1, 8, 128),
        # a user's own layer: odd sizes everywhere, codes as learnt, not packed
        _conv("conv5x5_ragged_b5", 5, 60, 37, 29, 150, 5, 1, 2, 6, 100, packed=False),
        # the reduced-precision table option on a layer that is in tolerance with it
        _conv("conv56_bf16_b8", 8, 64, 56, 56, 64, 3, 1, 1, 4, 128, lut="bf16", relu=False),
        # the whole network for one image
        {"name": "alexnet_b1", "op": "net", "N": 1},
        # the whole network at the throughput batch: the largest call
        {"name": "alexnet_b128", "op": "net", "N": 128},
        # encoding: AlexNet conv3's dense kernels to codebooks and codes, 10 rounds
        {"name": "kmeans_conv3", "op": "kmeans", "Ct": 384, "Cs": 256, "k": 3, "Csp": 4, "K": 128,
         "iters": 10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fc", "fc", "conv", "conv", "conv", "conv", "strided", "net", "kmeans"])
    if kind == "net":
        return {"op": "net", "N": _log(rng, 1, 128)}
    if kind == "kmeans":
        Csp = rng.choice([3, 4, 6, 8])
        return {"op": "kmeans", "Ct": rng.randint(64, 512), "Cs": Csp * rng.randint(8, 64),
                "k": rng.choice([1, 3, 5]), "Csp": Csp, "K": rng.choice([32, 64, 128, 256]),
                "iters": rng.randint(3, 10)}
    if kind == "fc":
        Csp = rng.choice([2, 3, 4, 4, 4, 8])
        return {"op": "fc", "N": _log(rng, 1, 256), "Cs": Csp * _log(rng, 64, 2304),
                "Ct": _log(rng, 100, 4096), "Csp": Csp, "K": rng.choice([16, 32, 32, 64, 128]),
                "bits": rng.random() < 0.3, "relu": rng.random() < 0.5}
    lut = "bf16" if rng.random() < 0.12 else "fp32"
    packed = rng.random() < 0.8
    while True:
        if kind == "strided":
            k, stride = rng.choice([(11, 4), (7, 2), (5, 2), (3, 2)])
            Csp, M = rng.choice([(3, 1), (4, rng.randint(1, 24)), (8, rng.randint(1, 16))])
            H, W, pad = rng.randint(27, 227), rng.randint(27, 227), rng.choice([0, k // 2])
        else:
            k, stride = rng.choice([1, 3, 3, 3, 5]), 1
            Csp = rng.choice([3, 4, 4, 4, 6, 8, 8])
            M, pad = _log(rng, 8, 512 // Csp), k // 2
            H = _log(rng, 7, 112)
            W = H if rng.random() < 0.6 else _log(rng, 7, 112)
        N, Ct, K = _log(rng, 1, 128), _log(rng, 32, 512), rng.choice([32, 64, 100, 128, 256])
        ho, wo = (H + 2 * pad - k) // stride + 1, (W + 2 * pad - k) // stride + 1
        # no more look-ups, table entries or bytes than a large single layer has
        if N * M * (ho * wo * Ct * k * k + H * W * K) <= 1e10 and \
                N * max(Csp * M * H * W, Ct * ho * wo) <= 1.5e8:
            return {"op": "conv", "N": N, "Cs": Csp * M, "H": H, "W": W, "Ct": Ct, "k": k,
                    "stride": stride, "pad": pad, "Csp": Csp, "K": K, "packed": packed,
                    "lut": lut, "relu": rng.random() < 0.5}


# ------------------------------------------------------------------ inputs
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1009 + salt)
    return g


def _normal(g, shape, std=1.0):
    return torch.randn(shape, generator=g, device="cuda") * std


def _codes(g, shape, K):
    return torch.randint(0, K, shape, generator=g, device="cuda", dtype=torch.uint8)


def _layer(g, M, K, Csp, codes_shape, fan_in, Ct):
    """Codebooks at He scale, codes uniform (no locality to profit from), biases."""
    D = _normal(g, (M, K, Csp), math.sqrt(2.0 / fan_in))
    return D, _codes(g, codes_shape, K), _normal(g, (Ct,), 0.1)


def _alex_layers(g):
    """[(kind, ..., D, codes, bias)] of the stack, canonical codes, and shapes."""
    c, h, w = ALEX_IN
    out = []
    for L in ALEX:
        if L[0] == "conv":
            _, ct, k, s, p, csp, K = L
            m = c // csp
            out.append((L, _layer(g, m, K, csp, (ct, k * k, m), k * k * c, ct), (c, h, w)))
            c, h, w = ct, (h + 2 * p - k) // s + 1, (w + 2 * p - k) // s + 1
        elif L[0] == "pool":
            out.append((L, None, (c, h, w)))
            h, w = (h - L[1]) // L[2] + 1, (w - L[1]) // L[2] + 1
        else:
            _, ct, csp, K, _ = L
            m = c * h * w // csp
            out.append((L, _layer(g, m, K, csp, (m, ct), c * h * w, ct), (c, h, w)))
            c, h, w = ct, 1, 1
    return out


def _data(case, seed):
    """The case's tensors as a user has them before any preparation."""
    op = case["op"]
    g = _gen(seed, {"fc": 1, "conv": 2, "net": 3, "kmeans": 4}[op])
    if op == "fc":
        M = case["Cs"] // case["Csp"]
        x = _normal(g, (case["N"], case["Cs"])).clamp_(min=0)  # follows a ReLU
        return (x,) + _layer(g, M, case["K"], case["Csp"], (M, case["Ct"]), case["Cs"], case["Ct"])
    if op == "conv":
        M, k = case["Cs"] // case["Csp"], case["k"]
        x = _normal(g, (case["N"], case["Cs"], case["H"], case["W"]))
        if case["Cs"] > 3:  # follows a ReLU; images do not
            x.clamp_(min=0)
        return (x,) + _layer(g, M, case["K"], case["Csp"], (case["Ct"], k * k, M),
                             k * k * case["Cs"], case["Ct"])
    if op == "net":
        return _normal(g, (case["N"],) + ALEX_IN), _alex_layers(g)
    # kmeans: dense kernels with a spread of scales, K of their sub-vectors as the start
    Ct, Cs, k, Csp, K = case["Ct"], case["Cs"], case["k"], case["Csp"], case["K"]
    W = _normal(g, (Ct, Cs, k, k), math.sqrt(2.0 / (k * k * Cs)))
    W *= torch.rand((Ct, 1, 1, 1), generator=g, device="cuda") + 0.5
    pts = W.view(Ct, Cs // Csp, Csp, k * k).permute(1, 0, 3, 2).reshape(Cs // Csp, -1, Csp)
    pick = torch.randint(0, pts.shape[1], (K,), generator=g, device="cuda")
    return W, pts[:, pick].contiguous()


def prepare(case, seed):
    op = case["op"]
    if op == "fc":
        x, D, codes, bias = _data(case, seed)
        if case["bits"]:
            codes = q.fc_pack_codes(codes, case["K"])
        return {"case": case, "x": x, "D": D, "codes": codes, "bias": bias}
    if op == "conv":
        x, D, codes, bias = _data(case, seed)
        if case["packed"]:
            codes = q.conv_pack_codes(codes, case["K"], case["k"], case["k"])
        return {"case": case, "x": x, "D": D, "codes": codes, "bias": bias}
    if op == "net":
        x, layers = _data(case, seed)
        built = []
        for L, p, _ in layers:
            if L[0] == "conv":
                D, codes, bias = p
                built.append(q.ConvLayer(D, q.conv_pack_codes(codes, L[6], L[2], L[2]), bias, L[1],
                                         L[2], L[2], L[3], L[4], True, packed=True))
            elif L[0] == "pool":
                built.append(q.PoolLayer(L[1], L[2]))
            else:
                built.append(q.FCLayer(p[0], p[1], p[2], L[4]))
        net = q.Net(built, ALEX_IN)
        return {"case": case, "x": x, "net": net, "workspace": net.alloc_workspace(case["N"])}
    W, init = _data(case, seed)
    return {"case": case, "W": W, "init": init}


def run(state):
    c = state["case"]
    if c["op"] == "fc":
        return q.fc_forward(state["x"], state["D"], state["codes"], state["bias"], relu=c["relu"],
                            Ct=c["Ct"])
    if c["op"] == "conv":
        return q.conv_forward(state["x"], state["D"], state["codes"], c["k"], c["k"], c["stride"],
                              c["pad"], state["bias"], relu=c["relu"], packed=c["packed"],
                              Ct=c["Ct"], lut=c["lut"])
    if c["op"] == "net":
        return state["net"].forward(state["x"], workspace=state["workspace"])
    return q.pq_quantize_conv(state["W"], c["Csp"], c["K"], state["init"], c["iters"])


# ------------------------------------------------------- what a pass must do
def _pq_work(N, Csp, K, M, positions, outputs, lookups_per_output):
    """flops of a layer's two stages: table entries (a dot product of C's
    terms each), then one add per look-up."""
    return N * (2.0 * positions * M * K * Csp + outputs * float(lookups_per_output))


def work(case):
    op = case["op"]
    if op == "fc":
        N, Cs, Ct, Csp, K = (case[k] for k in ("N", "Cs", "Ct", "Csp", "K"))
        M = Cs // Csp
        code_bytes = M * Ct * (math.ceil(math.log2(K)) / 8 if case["bits"] else 1)
        return {"bytes": 4 * (N * Cs + M * K * Csp + Ct + N * Ct) + code_bytes,
                "flops": _pq_work(N, Csp, K, M, 1, Ct, M)}
    if op == "conv":
        N, Cs, H, W, Ct, k, Csp, K = (case[n] for n in ("N", "Cs", "H", "W", "Ct", "k", "Csp", "K"))
        M = Cs // Csp
        ho = (H + 2 * case["pad"] - k) // case["stride"] + 1
        wo = (W + 2 * case["pad"] - k) // case["stride"] + 1
        return {"bytes": 4 * (N * Cs * H * W + M * K * Csp + Ct + N * Ct * ho * wo) + Ct * k * k * M,
                "flops": _pq_work(N, Csp, K, M, H * W, Ct * ho * wo, k * k * M)}
    if op == "net":
        N = case["N"]
        c, h, w = ALEX_IN
        nbytes, flops = 4.0 * N * (c * h * w + 1000), 0.0
        for L in ALEX:
            if L[0] == "conv":
                _, ct, k, s, p, csp, K = L
                m, ho, wo = c // csp, (h + 2 * p - k) // s + 1, (w + 2 * p - k) // s + 1
                nbytes += 4 * (m * K * csp + ct) + ct * k * k * m
                flops += _pq_work(N, csp, K, m, h * w, ct * ho * wo, k * k * m)
                c, h, w = ct, ho, wo
            elif L[0] == "pool":
                h, w = (h - L[1]) // L[2] + 1, (w - L[1]) // L[2] + 1
            else:
                _, ct, csp, K, _ = L
                m = c * h * w // csp
                nbytes += 4 * (m * K * csp + ct) + m * ct
                flops += _pq_work(N, csp, K, m, 1, ct, m)
                c, h, w = ct, 1, 1
        return {"bytes": nbytes, "flops": flops}
    Ct, Cs, k, Csp, K = (case[n] for n in ("Ct", "Cs", "k", "Csp", "K"))
    M, P = Cs // Csp, Ct * k * k
    return {"bytes": 4 * (Ct * Cs * k * k + 2 * M * K * Csp) + M * P,
            "flops": 3.0 * (case["iters"] + 1) * M * P * K * Csp}


# --------------------------------------------------- the same in 64 bits
def _conv64(x, D, codes, bias, k, stride, pad, relu):
    """Dense convolution with the kernels that the codes stand for, in float64."""
    M, K, Csp = D.shape
    Ct = codes.shape[0]
    W = D.double()[torch.arange(M, device=D.device)[None, None, :], codes.long()]  # [Ct, kk, M, C's]
    W = W.permute(0, 2, 3, 1).reshape(Ct, M * Csp, k, k)
    y = torch.cat([F.conv2d(x[i:i + 8].double(), W, bias.double(), stride=stride, padding=pad)
                   for i in range(0, x.shape[0], 8)])
    return y.relu_() if relu else y


def _fc64(x, D, codes, bias, relu):
    M, K, Csp = D.shape
    y = bias.double().repeat(x.shape[0], 1)
    m0, step = 0, max(1, (1 << 24) // (codes.shape[1] * Csp))
    while m0 < M:  # a slice of the sub-spaces at a time: the dense weights are large
        m1 = min(M, m0 + step)
        W = D[m0:m1].double()[torch.arange(m1 - m0, device=D.device)[:, None], codes[m0:m1].long()]
        y += x[:, m0 * Csp:m1 * Csp].double() @ W.transpose(1, 2).reshape(-1, codes.shape[1])
        m0 = m1
    return y.relu_() if relu else y


def exact(case, seed):
    op = case["op"]
    if op == "kmeans":
        return None  # which centroid is nearest is decided in 32 bits by definition here
    if op == "fc":
        x, D, codes, bias = _data(case, seed)
        return _fc64(x, D, codes, bias, case["relu"])
    if op == "conv":
        x, D, codes, bias = _data(case, seed)
        return _conv64(x, D, codes, bias, case["k"], case["stride"], case["pad"], case["relu"])
    x, layers = _data(case, seed)
    h = x.double()
    for L, p, _ in layers:
        if L[0] == "conv":
            h = _conv64(h, *p, L[2], L[3], L[4], True)
        elif L[0] == "pool":
            h = F.max_pool2d(h, L[1], L[2])
        else:
            h = _fc64(h.reshape(h.shape[0], -1), *p, L[4])
    return h
