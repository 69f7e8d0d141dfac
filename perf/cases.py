"""What the shift operators are measured on: the calls a user of the library makes, through its public entry points.

Sizes are those of the library's own configurations (ResNet18 / ResNet50 / VGG16 layers, the FC shapes of bench.py) or generic.  Inputs are drawn on
the GPU from the seed alone: int32 Q16.16 activations, signs with P(0) = 0.1, shifts uniform in [-15, 0] or two-sided geometric around a centre.
"""
from __future__ import annotations

import math

import torch

import paper_1905_13298_gb300 as ds
from paper_1905_13298_gb300 import networks

DEV = "cuda"


def listed():
    return [
        # the classifier of a network that answers one image at a time: the smallest call, all latency
        dict(name="fc_head_batch1", kind="fc", M=1, K=512, N=1000, bits=18, signed=False, centre=-9, relu=False, expand=True),
        # one FC layer of an MNIST-sized multi-layer perceptron, codes kept in the 6-bit blob
        dict(name="fc_64x784x512", kind="fc", M=64, K=784, N=512, bits=20, signed=False, centre=1, relu=False, expand=False),
        # VGG16's first FC layer at batch 64: many weights, few rows
        dict(name="fc_vgg16_fc1_batch64", kind="fc", M=64, K=25088, N=4096, bits=20, signed=False, centre=-11, relu=True, expand=True),
        # a token-parallel FC layer: the large dense contraction, signed activations
        dict(name="fc_8192x4096x4096", kind="fc", M=8192, K=4096, N=4096, bits=20, signed=True, centre=1, relu=False, expand=True),
        # the same layer on bf16 activations (the float variant)
        dict(name="fc_bf16_8192x4096x4096", kind="fc_bf16", M=8192, K=4096, N=4096, centre=1, relu=False),
        # the layer ResNet18 spends most of its time in, with its residual join
        dict(name="conv3x3_64x56x56_batch32", kind="conv", B=32, C=64, H=56, W=56, K=64, R=3, stride=1, pad=1, bits=20, signed=False, centre=-6, relu=True, residual=True, expand=True),
        # a strided layer on a small map: 49 output pixels per image
        dict(name="conv3x3s2_256x14x14_512", kind="conv", B=32, C=256, H=14, W=14, K=512, R=3, stride=2, pad=1, bits=18, signed=False, centre=-10, relu=True, residual=False, expand=True),
        # a ResNet50 bottleneck's 1x1 layer, codes kept in the 6-bit blob
        dict(name="conv1x1_1024x14x14_256", kind="conv", B=64, C=1024, H=14, W=14, K=256, R=1, stride=1, pad=0, bits=18, signed=False, centre=-9, relu=True, residual=False, expand=False),
        # the input gradient of a strided layer: four tap phases
        dict(name="conv3x3s2_backward_128x28", kind="conv_bwd", B=32, C=128, H=28, W=28, K=256, R=3, stride=2, pad=1, bits=18, centre=-9, expand=True),
        # a float model's layer made ready: quantized to codes, then packed
        dict(name="quantize_pack_4096x4096", kind="convert", N=4096, K=4096),
        # whole networks: the chained forward, for one image and for a batch
        dict(name="resnet18_batch1", kind="net", arch="resnet18", B=1, size=224),
        dict(name="resnet18_batch32", kind="net", arch="resnet18", B=32, size=224),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["fc", "fc", "fc", "conv", "conv", "conv", "conv", "conv_bwd", "fc_bf16", "convert", "net"])
    bits, expand, relu = rng.randint(14, 20), rng.random() < 0.6, rng.random() < 0.5
    if kind in ("fc", "fc_bf16"):
        while True:
            M, K, N = _log(rng, 1, 8192), _log(rng, 48, 25088), _log(rng, 10, 4096)
            if kind == "fc_bf16":
                K = (K + 7) // 8 * 8
            if M * K * N <= 2 ** 37 and K * N <= 2 ** 27 and M * K <= 2 ** 26:
                break
        centre = rng.choice([1, _centre(K)])
        if kind == "fc_bf16":
            return dict(kind=kind, M=M, K=K, N=N, centre=centre, relu=relu)
        return dict(kind=kind, M=M, K=K, N=N, bits=bits, signed=rng.random() < 0.5, centre=centre, relu=relu, expand=expand)
    if kind in ("conv", "conv_bwd"):
        while True:
            R, stride = rng.choice([1, 3, 3, 5, 7]), rng.choice([1, 1, 2])
            B, H, C, K = _log(rng, 1, 64), _log(rng, 7, 224), _log(rng, 3, 2048), _log(rng, 16, 2048)
            W = H + rng.choice([0, 0, 0, 1, -1, 5])
            if B * H * W * C * K * R * R <= 2 ** 35 * stride * stride and B * C * H * W <= 2 ** 27 and B * K * H * W <= 2 ** 27 * stride * stride and C * K * R * R <= 2 ** 25:
                break
        case = dict(kind=kind, B=B, C=C, H=H, W=W, K=K, R=R, stride=stride, pad=R // 2, bits=bits, centre=_centre((C if kind == "conv" else K) * R * R), expand=expand)
        if kind == "conv":
            case.update(signed=rng.random() < 0.3, relu=relu, residual=rng.random() < 0.3)
        return case
    if kind == "convert":
        return dict(kind=kind, N=_log(rng, 16, 4096), K=_log(rng, 48, 16384))
    return dict(kind=kind, arch=rng.choice(["resnet18", "resnet18", "resnet50"]), B=_log(rng, 1, 16), size=rng.choice([64, 96, 128, 160, 192, 224]))


def _centre(fan_in):
    """The shift centre that keeps a layer's output in its input's range."""
    return -round(math.log2(fan_in) / 2) - 4


def _gen(seed):
    return torch.Generator(DEV).manual_seed(seed * 7919 + 17)


def _codes(g, shape, centre):
    """Sign and shift codes: shifts uniform in [-15, 0] (centre 1) or centre + Geometric(1/2) - Geometric(1/2), clipped."""
    n = math.prod(shape)
    t = torch.rand(n, device=DEV, generator=g)
    s = torch.where(t < 0.1, 0, torch.where(t < 0.55, -1, 1))
    if centre > 0:
        p = torch.randint(-15, 1, (n,), device=DEV, generator=g)
    else:
        up, down = (torch.empty(n, device=DEV).geometric_(0.5, generator=g) for _ in range(2))
        p = (centre + up - down).clamp_(-15, 0)
    return s.to(torch.int8).reshape(shape), p.to(torch.int8).reshape(shape)


def _activations(g, shape, bits, signed):
    return torch.randint(-(1 << bits) if signed else 0, 1 << bits, shape, device=DEV, generator=g, dtype=torch.int32)


def _bias(g, n):
    return torch.randint(-(1 << 16), 1 << 16, (n,), device=DEV, generator=g, dtype=torch.int32)


def _out(case):
    f = lambda n: (n + 2 * case["pad"] - case["R"]) // case["stride"] + 1  # noqa: E731
    return f(case["H"]), f(case["W"])


def _inputs(case, seed):
    """The plain tensors of a layer's call."""
    g, kind = _gen(seed), case["kind"]
    d = {}
    if kind in ("fc", "fc_bf16"):
        M, K, N = case["M"], case["K"], case["N"]
        d["s"], d["p"] = _codes(g, (N, K), case["centre"])
        if kind == "fc":
            d["x"], d["b"] = _activations(g, (M, K), case["bits"], case["signed"]), _bias(g, N)
        else:
            d["x"] = torch.randn(M, K, device=DEV, generator=g).to(torch.bfloat16)
            d["b"] = torch.randn(N, device=DEV, generator=g)
    elif kind in ("conv", "conv_bwd"):
        B, C, K, R, (OH, OW) = case["B"], case["C"], case["K"], case["R"], _out(case)
        d["s"], d["p"] = _codes(g, (K, C, R, R), case["centre"])
        if kind == "conv":
            d["x"], d["b"] = _activations(g, (B, C, case["H"], case["W"]), case["bits"], case["signed"]), _bias(g, K)
            d["res"] = _activations(g, (B, K, OH, OW), case["bits"], False) if case["residual"] else None
        else:
            d["dy"] = _activations(g, (B, K, OH, OW), case["bits"], True)
    else:  # convert: log-uniform magnitudes across the shift range, both signs
        e = torch.rand(case["N"], case["K"], device=DEV, generator=g) * 18 - 17
        d["w"] = torch.exp2(e) * torch.where(torch.rand(e.shape, device=DEV, generator=g) < 0.5, -1.0, 1.0)
    return d


def _program(case):
    return networks.resnet_program(case["arch"], case["size"], case["size"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "net":
        g = _gen(seed)
        specs, shapes = _program(case)
        params = []
        for shape in shapes:
            s, p = _codes(g, shape, _centre(math.prod(shape[1:])))
            params.append((s.cpu().numpy(), p.cpu().numpy(), _bias(g, shape[0]).cpu().numpy()))
        net = networks.ShiftNetwork(specs, params, case["B"])
        return dict(kind=kind, net=net, x=_activations(g, (case["B"], 3, case["size"], case["size"]), 17, True))
    d = _inputs(case, seed)
    if kind == "convert":
        return dict(kind=kind, w=d["w"])
    s, p = d.pop("s"), d.pop("p")
    if kind == "fc_bf16":
        d["w"] = ds.expand_shift_weights_bf16(ds.pack_shift_weights(s, p))
    elif kind == "conv_bwd":
        d["w"] = ds.pack_shift_weights_backward(s, p, (case["stride"],) * 2, expand=case["expand"])
        d["shape"] = (case["B"], case["C"], case["H"], case["W"])
    else:
        d["w"] = ds.pack_shift_weights(s, p, expand=case["expand"])
    return dict(d, kind=kind, case=dict(case), amax=torch.zeros(2, dtype=torch.int32, device=DEV))


def run(state):
    kind = state["kind"]
    if kind == "net":
        return state["net"].forward(state["x"])
    if kind == "convert":
        s, p = ds.quantize_shift_weights(state["w"])
        w = ds.pack_shift_weights(s, p)
        return s, p, w.blob
    c = state["case"]
    if kind == "fc":
        return ds.linear_shift(state["x"], state["w"], state["b"], relu=c["relu"], amax_io=state["amax"])
    if kind == "fc_bf16":
        return ds.linear_shift_bf16(state["x"], state["w"], state["b"], relu=c["relu"])
    st, pd, R = c["stride"], c["pad"], c["R"]
    if kind == "conv":
        return ds.conv2d_shift(state["x"], state["w"], (R, R), state["b"], (st, st), (pd, pd), relu=c["relu"], residual=state["res"], amax_io=state["amax"])
    B, C, H, W = state["shape"]
    dx = torch.empty(state["shape"], dtype=torch.int32, device=DEV)
    ds.ds_conv2d_shift_backward_x(state["dy"], state["w"].desc, dx, B, C, H, W, c["K"], R, R, st, st, pd, pd, 0, state["amax"])
    return dx


def work(case):
    """Tensors read and written once, codes at the 6 bits of the blob; one shift and one add per term (two flops per term on bf16)."""
    kind = case["kind"]
    if kind in ("fc", "fc_bf16"):
        M, K, N = case["M"], case["K"], case["N"]
        codes, x = (2, 2) if kind == "fc_bf16" else (0.75, 4)
        return dict(bytes=M * K * x + N * K * codes + 4 * N + 4 * M * N, flops=2 * M * K * N)
    if kind in ("conv", "conv_bwd"):
        B, C, K, R, (OH, OW) = case["B"], case["C"], case["K"], case["R"], _out(case)
        x, y, w = B * C * case["H"] * case["W"], B * K * OH * OW, K * C * R * R
        return dict(bytes=4 * x + (8 if case.get("residual") else 4) * y + 0.75 * w + 4 * K, flops=2 * y * C * R * R)
    if kind == "convert":
        n = case["N"] * case["K"]
        return dict(bytes=n * (4 + 2 + 0.75), flops=2 * n)
    specs, shapes = _program(case)
    tensors = sum(math.prod(networks.output_shape(sp)) for sp in specs)
    terms = networks.shift_terms(specs, case["B"])
    return dict(bytes=4 * case["B"] * (3 * case["size"] ** 2 + 2 * tensors) + 0.75 * sum(math.prod(sh) for sh in shapes), flops=2 * terms)


def _shift_sum(x, s, p, product):
    """sum over the shift values k of product(x >> k, s where p == -k), exact in float64 (every sum is below 2^53)."""
    acc = None
    for k in range(16):
        w = torch.where(p == -k, s, torch.zeros_like(s))
        if bool((w != 0).any()):
            t = product((x >> k).double(), w.double())
            acc = t if acc is None else acc.add_(t)
    return acc


def _finish(acc, bias, residual, relu):
    if bias is not None:
        acc = acc + bias
    acc = acc.clamp_(-2.0 ** 31, 2.0 ** 31 - 1)
    if residual is not None:
        acc = (acc + residual).clamp_(-2.0 ** 31, 2.0 ** 31 - 1)
    return (acc.clamp_(min=0) if relu else acc).to(torch.int64)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("net", "convert") or work(case)["flops"] > 3e11:
        return None  # whole numbers and bytes throughout, held equal as they are; or too long in 64 bits
    d = _inputs(case, seed)
    if kind == "fc":
        acc = _shift_sum(d["x"], d["s"], d["p"], lambda a, w: a @ w.t())
        return _finish(acc, d["b"][None, :], None, case["relu"])
    if kind == "fc_bf16":
        y = d["x"].double() @ (d["s"].double() * torch.exp2(d["p"].double())).t() + d["b"].double()
        return y.clamp_(min=0) if case["relu"] else y
    B, C, K, R, st, (OH, OW) = case["B"], case["C"], case["K"], case["R"], case["stride"], _out(case)
    if kind == "conv":
        xp = torch.nn.functional.pad(d["x"], (case["pad"],) * 4)

        def conv(a, w):
            y = torch.zeros(K, B * OH * OW, dtype=torch.float64, device=DEV)
            for r in range(R):
                for q in range(R):
                    t = a[:, :, r:r + st * (OH - 1) + 1:st, q:q + st * (OW - 1) + 1:st]
                    y.addmm_(w[:, :, r, q], t.transpose(0, 1).reshape(C, -1))
            return y

        acc = _shift_sum(xp, d["s"], d["p"], conv).reshape(K, B, OH, OW).transpose(0, 1)
        return _finish(acc, d["b"][None, :, None, None], d["res"], case["relu"])

    def grad(a, w):
        dx = torch.zeros(C, B, case["H"] + 2 * case["pad"], case["W"] + 2 * case["pad"], dtype=torch.float64, device=DEV)
        a = a.transpose(0, 1).reshape(K, -1)
        for r in range(R):
            for q in range(R):
                dx[:, :, r:r + st * (OH - 1) + 1:st, q:q + st * (OW - 1) + 1:st] += (w[:, :, r, q].t() @ a).reshape(C, B, OH, OW)
        return dx

    acc, pd = _shift_sum(d["dy"], d["s"], d["p"], grad), case["pad"]
    return _finish(acc[:, :, pd:pd + case["H"], pd:pd + case["W"]].transpose(0, 1), None, None, False)
