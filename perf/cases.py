"""The work that a user of this framework has it do, as cases that can be timed and compared.

A case is a dict of plain values.  ``kind`` says which entry point it calls:

  product   ``linear`` (fp32 output) or, with ``out`` or ``bias`` set, ``linear_fused``
  conv      ``conv2d`` (NHWC, fp32 output) or, with ``out`` or ``bias`` set, ``conv2d_fused``
  stack     the 52 convolutions of ResNet-50 after the stem, chained through ``conv2d_fused``
  pack      ``pack`` of dense weights
  dropout   ``td_mask``, one targeted-dropout step of a training pass

What a program holds before the call (packed weights, biases, status words, the buffers of a whole
network) is made by ``prepare``; every pass starts from packed weights, so the weights' expansion is
part of each product.  Inputs are seeded draws with the distributions of ``workloads.py``: He-normal
weights, ReLU(N(0, 1)) activations behind a ReLU, N(0, 1) or U(-1, 1) elsewhere.
"""
import math

import torch

import paper_1910_11971_gb300 as cci
from paper_1910_11971_gb300 import workloads as wl

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
# (G, K) of the paper's networks and of the sweep
GROUPS = ((4, 1), (4, 2), (8, 1), (8, 2), (8, 4), (16, 1), (16, 2), (16, 4), (16, 8), (32, 4), (32, 8))


def _product(name, N, Cin, Cout, G, K, dtype, x="relu_normal", bias=False, relu=False, out=""):
    return {"name": name, "kind": "product", "N": N, "Cin": Cin, "Cout": Cout, "G": G, "K": K, "dtype": dtype, "x": x,
            "bias": bias, "relu": relu, "out": out}


def _conv(name, B, H, W, Cin, Cout, k, stride, pad, G, K, dtype, bias=False, relu=False, out=""):
    return {"name": name, "kind": "conv", "B": B, "H": H, "W": W, "Cin": Cin, "Cout": Cout, "k": k, "stride": stride,
            "pad": pad, "G": G, "K": K, "dtype": dtype, "bias": bias, "relu": relu, "out": out}


def listed():
    return [
        # the smallest call: a 64 -> 64 layer on 32 columns, where launches and latency are all there is
        _product("product_tiny_f32", 32, 64, 64, 4, 2, "f32", x="uniform"),
        # a request of a few columns through a wide layer: serving, where the packed weights are what is read
        _product("product_serve", 16, 4096, 4096, 8, 2, "bf16", x="normal", bias=True, relu=True, out="bf16"),
        # a classifier head on a batch that is no multiple of a tile: 2048 -> 1000 with bias, fp32 logits
        _product("product_head", 100, 2048, 1000, 8, 2, "bf16", bias=True, out="f32"),
        # the benchmark's headline point: a large product, bf16
        _product("product_sweep_4096", 8192, 4096, 4096, 8, 2, "bf16", x="normal"),
        # a ResNet bottleneck 1x1 on 32 images in fp32
        _product("bottleneck_1x1_f32", 100352, 256, 1024, 8, 2, "f32"),
        # 3x3 convolution, 28 x 28, 128 -> 128, fp32 output
        _conv("conv3x3_28", 64, 28, 28, 128, 128, 3, 1, 1, 16, 4, "bf16"),
        # ResNet-50's widest-image 3x3 layer at batch 128, bias, ReLU and bf16 output as inside a network
        _conv("conv3x3_56_fused", 128, 56, 56, 64, 64, 3, 1, 1, 8, 2, "bf16", bias=True, relu=True, out="bf16"),
        # a strided 3x3 layer (28 x 28 -> 14 x 14) of the same network
        _conv("conv3x3_s2_fused", 128, 28, 28, 256, 256, 3, 2, 1, 8, 2, "bf16", bias=True, relu=True, out="bf16"),
        # MobileNetV2's first expansion: a pointwise layer of 16 input channels on 1.6 M pixels
        _conv("pointwise_112_fused", 128, 112, 112, 16, 96, 1, 1, 0, 8, 2, "bf16", bias=True, relu=True, out="bf16"),
        # a whole network's convolutions, one after the other, at a serving batch
        {"name": "resnet50_stack", "kind": "stack", "B": 32, "G": 8, "K": 2},
        # compressing a wide layer's weights
        {"name": "pack_4096", "kind": "pack", "Cout": 4096, "R": 4096, "G": 8, "K": 2, "dtype": "bf16"},
        # the mask step of training on the fp32 weights of a wide layer
        {"name": "dropout_4096", "kind": "dropout", "Cout": 4096, "R": 4096, "G": 16, "K": 2, "dtype": "f32", "rate": 0.75},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo, hi, multiple):
    return max(1, _log_int(rng, lo, hi) // multiple) * multiple


def draw(rng):
    """One more case of the same ranges: any number of columns or pixels, channel counts in multiples of
    the 16-byte vectors that the layers are laid out in, every (G, K) of the paper's networks."""
    G, K = rng.choice(GROUPS)
    kind = rng.choice(("product", "product", "product", "conv", "conv", "conv", "stack", "pack", "dropout"))
    dtype = rng.choice(("bf16", "bf16", "f32"))
    unit = 8 if dtype == "bf16" else 4
    fused = rng.random() < 0.5
    ep = {"bias": fused, "relu": fused and rng.random() < 0.7,
          "out": rng.choice(("bf16", "f32")) if fused else ""}
    if kind == "product":
        Cin = _channels(rng, 16, 4096, unit)
        Cout = _channels(rng, 32, 4096, max(G, 8))
        # at most the sweep's work; fp32 layers at most the bottleneck's
        most = 8192 * 4096 * 4096 if dtype == "bf16" else 100352 * 256 * 1024
        N = _log_int(rng, 1, min(8192 if rng.random() < 0.5 else 100352, max(1, most // (Cin * Cout))))
        return {"kind": kind, "N": N, "Cin": Cin, "Cout": Cout, "G": G, "K": K, "dtype": dtype,
                "x": rng.choice(("relu_normal", "normal", "uniform")), **ep}
    if kind == "conv":
        H = _log_int(rng, 7, 56)
        W = H if rng.random() < 0.6 else _log_int(rng, 7, 56)
        Cin = _channels(rng, 16, 512, rng.choice((unit, 32, 64)))
        Cout = _channels(rng, 32, 512, max(G, 8))
        k = rng.choice((1, 3, 3))
        stride = rng.choice((1, 1, 2))
        # the work of 128 images of a ResNet layer in bf16, a fifth of it in fp32
        most = (128 if dtype == "bf16" else 25) * 56 * 56 * 64 * 64 * 9
        per = ((H - 1) // stride + 1) * ((W - 1) // stride + 1) * Cin * Cout * k * k
        return {"kind": kind, "B": _log_int(rng, 1, min(128, max(1, most // per))), "H": H, "W": W, "Cin": Cin,
                "Cout": Cout, "k": k, "stride": stride, "pad": k // 2, "G": G, "K": K, "dtype": dtype, **ep}
    if kind == "stack":
        return {"kind": kind, "B": _log_int(rng, 1, 32), "G": 8, "K": rng.choice((1, 2, 4))}
    if kind == "pack":
        return {"kind": kind, "Cout": _channels(rng, 64, 4096, G), "R": _log_int(rng, 64, 4096), "G": G, "K": K,
                "dtype": dtype}
    return {"kind": kind, "Cout": _channels(rng, 64, 4096, G), "R": _log_int(rng, 64, 4096), "G": G, "K": K,
            "dtype": dtype, "rate": rng.choice((0.5, 0.75, 1.0))}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1009 + stream)
    return g


def _normal(shape, std, dtype, seed, stream):
    return (torch.randn(shape, generator=_gen(seed, stream), device="cuda") * std).to(DTYPES[dtype])


def _activations(shape, dist, dtype, seed):
    g = _gen(seed, 1)
    if dist == "uniform":
        t = torch.rand(shape, generator=g, device="cuda") * 2.0 - 1.0
    else:
        t = torch.randn(shape, generator=g, device="cuda")
        if dist == "relu_normal":
            t.clamp_min_(0.0)
    return t.to(DTYPES[dtype])


def _layer(case, seed):
    """(X, W, bias) of a product or a convolution; W is [Cout][R]."""
    if case["kind"] == "product":
        R = case["Cin"]
        X = _activations((case["N"], R), case["x"], case["dtype"], seed)
    else:
        R = case["k"] * case["k"] * case["Cin"]
        X = _activations((case["B"], case["H"], case["W"], case["Cin"]), "relu_normal", case["dtype"], seed)
    W = _normal((case["Cout"], R), math.sqrt(2.0 / R), case["dtype"], seed, 2)
    bias = _normal((case["Cout"],), 0.1, "f32", seed, 3) if case["bias"] else None
    return X, W, bias


def _stack(case, seed):
    """[(layer, role, W, bias)] and the first block's input."""
    layers = wl.resnet50_layers(batch=case["B"], G=case["G"], K=case["K"])
    every = []
    for i, (c, role) in enumerate(zip(layers, wl.resnet50_roles())):
        every.append((c, role, _normal((c.Cout, c.R), c.w_std, "bf16", seed, 10 + 2 * i),
                      _normal((c.Cout,), 0.1, "f32", seed, 11 + 2 * i)))
    c = layers[0]
    return every, _activations((c.B, c.H, c.W, c.Cin), "relu_normal", "bf16", seed)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("pack", "dropout"):
        W = _normal((case["Cout"], case["R"]), math.sqrt(2.0 / case["R"]), case["dtype"], seed, 2)
        status = cci.new_status(W.device)
        if kind == "pack":
            return {"case": case, "W": W, "status": status}
        u = torch.rand((case["Cout"], case["R"]), generator=_gen(seed, 4), device="cuda")
        return {"case": case, "W": W, "u": u, "status": status}
    if kind == "stack":
        every, x = _stack(case, seed)
        calls, most = [], 0
        for c, role, W, bias in every:
            v, i = cci.pack(W, c.G, c.K, check=False)
            out = torch.empty((c.B, c.P, c.Q, c.Cout), dtype=torch.bfloat16, device="cuda")
            most = max(most, cci.workspace_size(cci.ALGO_AUTO, torch.bfloat16, c.Cout, c.R))
            calls.append((c, role, v, i, bias, out))
        # one workspace for the whole network: its layers run one after the other
        return {"case": case, "x": x, "calls": calls, "ws": torch.empty(most, dtype=torch.uint8, device="cuda")}
    X, W, bias = _layer(case, seed)
    v, i = cci.pack(W, case["G"], case["K"], check=False)
    return {"case": case, "X": X, "v": v, "i": i, "bias": bias}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "pack":
        return cci.pack(state["W"], case["G"], case["K"], status=state["status"], check=False)
    if kind == "dropout":
        return cci.td_mask(state["W"], case["G"], case["K"], case["rate"], state["u"], status=state["status"])
    if kind == "stack":
        block, prev, pending, stages = state["x"], None, None, []
        for c, role, v, i, bias, out in state["calls"]:
            if role == "a" and pending is not None:  # a new block reads the last block's output
                if pending.shape[1] != c.P:
                    stages.append(pending)
                block, pending = pending, None
            src = block if role in ("a", "proj") else prev
            cci.conv2d_fused(src, v, i, c.Cout, c.G, c.K, c.KH, c.KW, (c.stride, c.stride), (c.pad, c.pad), bias=bias,
                             relu=role in ("a", "b"), out=out, workspace=state["ws"])
            if role in ("a", "b"):
                prev = out
            elif role == "c":
                pending = out
            else:
                stages.append(out)
        return stages + [pending]
    fused = case["bias"] or case["out"] != ""
    args = (state["X"], state["v"], state["i"], case["Cout"], case["G"], case["K"])
    more = {"bias": state["bias"], "relu": case["relu"], "out_dtype": DTYPES[case["out"] or "f32"]} if fused else {}
    if kind == "product":
        return cci.linear_fused(*args, **more) if fused else cci.linear(*args)
    geo = (case["k"], case["k"], (case["stride"],) * 2, (case["pad"],) * 2)
    return cci.conv2d_fused(*args, *geo, **more) if fused else cci.conv2d(*args, *geo)


# ---------------------------------------------------------------------------
# work, tolerances and the results in 64 bits
# ---------------------------------------------------------------------------

def _layer_work(N, x_elems, R, Cout, G, K, elem, out_elem, bias):
    packed = Cout // G * R * K * (elem + 1)
    return {"bytes": x_elems * elem + packed + N * Cout * out_elem + (Cout * 4 if bias else 0),
            "flops": 2 * N * R * Cout * K // G}


def work(case):
    kind = case["kind"]
    if kind in ("pack", "dropout"):
        elem = 4 if case["dtype"] == "f32" else 2
        n = case["Cout"] * case["R"]
        if kind == "pack":
            return {"bytes": n * elem + n // case["G"] * case["K"] * (elem + 1), "flops": 0}
        return {"bytes": n * (elem + 4 + elem + 1), "flops": 0}
    if kind == "stack":
        total = {"bytes": 0, "flops": 0}
        for c in wl.resnet50_layers(batch=case["B"], G=case["G"], K=case["K"]):
            w = _layer_work(c.N, c.B * c.H * c.W * c.Cin, c.R, c.Cout, c.G, c.K, 2, 2, True)
            total = {k: total[k] + w[k] for k in total}
        return total
    elem = 4 if case["dtype"] == "f32" else 2
    out_elem = 2 if case["out"] == "bf16" else 4
    if kind == "product":
        N, R = case["N"], case["Cin"]
        x = N * R
    else:
        P, Q = ((case[s] + 2 * case["pad"] - case["k"]) // case["stride"] + 1 for s in ("H", "W"))
        N, R = case["B"] * P * Q, case["k"] * case["k"] * case["Cin"]
        x = case["B"] * case["H"] * case["W"] * case["Cin"]
    return _layer_work(N, x, R, case["Cout"], case["G"], case["K"], elem, out_elem, case["bias"])


def tolerance(case):
    kind = case["kind"]
    if kind in ("pack", "dropout"):
        return "exact"
    if kind == "stack":
        # bf16 between 52 layers: a change of the sum's order in one of them moves roundings in all that follow
        return {"rel": 2e-2, "max": 0.3}
    if case["out"] == "bf16":
        return {"rel": 7e-3, "max": 3e-2}  # one rounding to bf16
    if case["dtype"] == "f32":
        return {"rel": 1.5e-5, "max": 3e-4}  # fp32 sums of the fp32 split (three terms of tf32 and bf16 operands)
    return {"rel": 5e-6, "max": 2e-4}  # fp32 sums of exact bf16 products


def _dense(W, G, K):
    """W [Cout][R] in 64 bits with all but the K largest |w| of each group zeroed (ties: the lower index), and the
    kept indices [Cout/G][K][R] in increasing order."""
    Cout, R = W.shape
    w = W.double().view(Cout // G, G, R)
    keep = torch.sort(w.abs(), dim=1, descending=True, stable=True).indices[:, :K].sort(dim=1).values
    mask = torch.zeros_like(w).scatter_(1, keep, 1.0)
    return (w * mask).view(Cout, R), keep, mask.view(Cout, R)


def _conv64(X, Wd, k, stride, pad, Cout):
    """NHWC convolution in 64 bits, one product per tap."""
    B, H, W, Cin = X.shape
    P, Q = (H + 2 * pad - k) // stride + 1, (W + 2 * pad - k) // stride + 1
    xp = torch.nn.functional.pad(X.double(), (0, 0, pad, pad, pad, pad))
    w = Wd.view(Cout, k, k, Cin)
    y = torch.zeros((B * P * Q, Cout), dtype=torch.float64, device=X.device)
    for kh in range(k):
        for kw in range(k):
            tap = xp[:, kh:kh + stride * (P - 1) + 1:stride, kw:kw + stride * (Q - 1) + 1:stride]
            y.addmm_(tap.reshape(-1, Cin), w[:, kh, kw].t())
    return y.view(B, P, Q, Cout)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("pack", "dropout"):
        W = _normal((case["Cout"], case["R"]), math.sqrt(2.0 / case["R"]), case["dtype"], seed, 2)
        G, K = case["G"], case["K"]
        _, keep, mask = _dense(W, G, K)
        if kind == "pack":
            v = W.double().view(case["Cout"] // G, G, case["R"]).gather(1, keep)
            return v.permute(0, 2, 1).contiguous(), keep.permute(0, 2, 1).contiguous().to(torch.uint8)
        u = torch.rand((case["Cout"], case["R"]), generator=_gen(seed, 4), device="cuda")
        kept = (mask > 0) | ~(u < case["rate"])
        return W.double() * kept, kept.to(torch.uint8)
    if kind == "stack":
        # activations are bf16 between the layers by definition: rounded there, all sums in 64 bits
        every, x = _stack(case, seed)
        block, prev, pending, stages = x.double(), None, None, []
        for c, role, W, bias in every:
            if role == "a" and pending is not None:
                if pending.shape[1] != c.P:
                    stages.append(pending)
                block, pending = pending, None
            src = block if role in ("a", "proj") else prev
            y = _conv64(src, _dense(W, c.G, c.K)[0], c.KH, c.stride, c.pad, c.Cout) + bias.double()
            if role in ("a", "b"):
                y.clamp_min_(0.0)
            y = y.to(torch.bfloat16).double()
            if role in ("a", "b"):
                prev = y
            elif role == "c":
                pending = y
            else:
                stages.append(y)
        return stages + [pending]
    X, W, bias = _layer(case, seed)
    Wd = _dense(W, case["G"], case["K"])[0]
    if kind == "product":
        y = X.double() @ Wd.t()
    else:
        y = _conv64(X, Wd, case["k"], case["stride"], case["pad"], case["Cout"])
    if bias is not None:
        y += bias.double()
    if case["relu"]:
        y.clamp_min_(0.0)
    return y
