"""Timed cases of the framework: what a user's program calls, over the sizes it calls it with.

Kinds of case, each through the public entry points of ``paper_2207_08820_b200``:

  conv        one quantised layer (``api.bitserial_conv2d``) on packed activations, with packed filters (``engine`` "popc") or
              filters prepared for the tensor cores ("tc", where ``api.tc_supported`` takes the shape); packed codes or
              int32 accumulators come out
  gemm        the matrix product of an im2col'ed layer or a fully connected one (``api.bitserial_gemm`` / ``bitserial_gemm_tc``)
  net         a stack of quantised layers (``net.BitserialNet``) on a float32 input, launched layer by layer ("forward") or as a
              captured graph whose input changes from pass to pass ("replay")
  classifier  the whole mixed-precision classifier (``net.BitserialFullNet``): images in, logits out
  pack        quantise and bit-pack a tensor (``api.bitpack_activations``), float32 values or int8 codes, both layouts

Inputs follow the repository's own recipe (``workloads.py``): codes uniform over their range, zero-mean weights with calibrated
scale and bias in layer stacks, float inputs whose codes are uniform, normalised images.  They are drawn on the GPU.
"""
import math

import numpy as np
import torch

from paper_2207_08820_b200 import api, net, workloads as wl

ACT_SCALE = 0.25
STACKS = {"resnet18_body": wl.resnet18_body, "resnet50_body": wl.resnet50_body, "vgg16_ssd_body": wl.vgg16_ssd_body,
          "detection_backbone": wl.detection_backbone}


# ------------------------------------------------------------------------------------------------------------- the cases

def listed():
    def conv(name, N, C, H, W, O, k, stride, a, w, engine, out="codes", residual=False):
        return dict(name=name, kind="conv", N=N, C=C, H=H, W=W, O=O, k=k, stride=stride, a_bits=a, w_bits=w, engine=engine,
                    out=out, residual=residual)

    def gemm(name, M, N, K, a, w, engine, out="acc"):
        return dict(name=name, kind="gemm", M=M, N=N, K=K, a_bits=a, w_bits=w, engine=engine, out=out)

    return [
        # one layer of a single image: the smallest call, all latency
        conv("layer 1x64x56x56 3x3", 1, 64, 56, 56, 64, 3, 1, 2, 2, "popc"),
        # the widest codes of the bit-width study, where the plane pairs are many and the arithmetic counts
        conv("layer 32x256x28x28 3x3 w3a3", 32, 256, 28, 28, 256, 3, 1, 3, 3, "popc"),
        # nothing divides anything: odd image, 80 filters, 1-bit activations under 2-bit weights, stride 2
        conv("layer 5x96x37x45 3x3 s2 w2a1", 5, 96, 37, 45, 80, 3, 2, 1, 2, "popc"),
        # matrix products of a small and of a middling layer, 1-bit weights
        gemm("product 256x256x576", 256, 256, 576, 2, 1, "popc"),
        gemm("product 1024x1024x2304", 1024, 1024, 2304, 2, 1, "popc"),
        # the largest product, its filters prepared once
        gemm("product 4096x4096x4608 tc", 4096, 4096, 4608, 2, 1, "tc"),
        # the residual stack: throughput at batch 64, and one image at a time as a captured graph
        dict(name="residual stack b64", kind="net", stack="resnet18_body", batch=64, hw=56, a_bits=2, w_bits=2, engine="tc", mode="forward"),
        dict(name="residual stack b1 graph", kind="net", stack="resnet18_body", batch=1, hw=56, a_bits=2, w_bits=2, engine="tc", mode="replay"),
        # detection: a large input, many 1x1 layers over few channels, concatenations
        dict(name="detection stack b16", kind="net", stack="detection_backbone", batch=16, hw=320, a_bits=2, w_bits=2, engine="tc", mode="forward"),
        # images in, logits out
        dict(name="classifier b64 224px", kind="classifier", batch=64, hw=224),
        # the quantiser in front of the residual stack, and codes that come from elsewhere with a ragged shape
        dict(name="pack 64x64x56x56 f32", kind="pack", N=64, C=64, H=56, W=56, bits=2, dtype="f32", layout="nchw"),
        dict(name="pack 48x50x45x61 i8 nhwc", kind="pack", N=48, C=50, H=45, W=61, bits=3, dtype="i8", layout="nhwc"),
    ]


def _spread(rng, lo, hi):
    """A whole number of [lo, hi], uniform over the logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        kind = rng.choice(["conv", "conv", "gemm", "gemm", "net", "net", "net", "classifier", "pack", "pack"])
        a, w = rng.choice([(2, 2), (2, 2), (2, 1), (1, 2), (1, 1), (3, 3), (2, 3), (4, 4)])
        engine = rng.choice(["popc", "tc"])
        if kind == "conv":
            c = 32 * _spread(rng, 1, 16) if rng.random() < 0.7 else _spread(rng, 16, 400)
            o = 32 * _spread(rng, 1, 16) if rng.random() < 0.7 else _spread(rng, 16, 400)
            h = _spread(rng, 7, 112)
            case = dict(kind=kind, N=_spread(rng, 1, 64), C=c, H=h, W=max(7, h + rng.randint(-3, 3)), O=o,
                        k=rng.choice([1, 3, 3, 3, 5]), stride=rng.choice([1, 1, 2]), a_bits=a, w_bits=w, engine=engine,
                        out=rng.choice(["codes", "codes", "acc"]), residual=rng.random() < 0.3)
        elif kind == "gemm":
            case = dict(kind=kind, M=_spread(rng, 100, 4096), N=_spread(rng, 64, 4096), K=64 * _spread(rng, 4, 72) if rng.random() < 0.7 else _spread(rng, 256, 4608),
                        a_bits=a, w_bits=w, engine=engine, out=rng.choice(["acc", "acc", "codes"]))
        elif kind == "net":
            stack = rng.choice(["resnet18_body", "resnet18_body", "resnet50_body", "vgg16_ssd_body", "detection_backbone"])
            lo, hi = {"resnet18_body": (28, 72), "resnet50_body": (28, 72), "vgg16_ssd_body": (64, 300), "detection_backbone": (64, 320)}[stack]
            hw = _spread(rng, lo, hi)
            if rng.random() < 0.5:
                hw -= hw % 4
            case = dict(kind=kind, stack=stack, batch=_spread(rng, 1, 64), hw=hw, a_bits=rng.choice([2, 2, 1]), w_bits=2, engine="tc",
                        mode=rng.choice(["forward", "forward", "replay"]))
        elif kind == "classifier":
            case = dict(kind=kind, batch=_spread(rng, 1, 64), hw=4 * rng.randint(40, 64))
        else:
            case = dict(kind=kind, N=_spread(rng, 1, 64), C=_spread(rng, 16, 512), H=_spread(rng, 7, 160), W=_spread(rng, 7, 160), bits=rng.choice([1, 2, 2, 3, 4]),
                        dtype=rng.choice(["f32", "f32", "i8"]), layout=rng.choice(["nchw", "nchw", "nhwc"]))
        # no more than the largest listed ones: 217 to 232 GFLOP in a stack, 266 G plane-pair operations in a single layer, 13 M values packed
        if case["kind"] in ("conv", "gemm"):
            if work(case)["flops"] * case["a_bits"] * case["w_bits"] > 266e9:
                continue
        elif case["kind"] in ("net", "classifier"):
            w_ = work(case)
            if w_["flops"] > 217e9 or w_["bytes"] > 250e6:
                continue
        elif case["N"] * case["C"] * case["H"] * case["W"] > 13e6 or case["N"] * case["C"] * case["H"] * case["W"] < 1e5:
            continue
        return case


# ---------------------------------------------------------------------------------------------------------------- inputs

def _codes(gen, shape, bits, sign):
    if sign == api.BIPOLAR:
        return torch.randint(0, 2, shape, generator=gen, device="cuda", dtype=torch.int8) * 2 - 1
    lo, hi = wl.code_range(bits, sign)
    return torch.randint(lo, hi + 1, shape, generator=gen, device="cuda", dtype=torch.int8)


def _zero_mean_weights(gen, shape, bits, sign):
    """The distribution of ``workloads.rand_weights_zero_mean`` (every filter sums to about zero)."""
    if sign != api.SIGNED or bits < 2:
        return _codes(gen, shape, bits, sign)
    lo, hi = wl.code_range(bits, sign)
    p = np.ones(hi - lo + 1)
    v = np.arange(lo, hi + 1)
    p[:2] = 0.5
    p[v > 0] *= -float((p * v)[v < 0].sum()) / float((p * v)[v > 0].sum())
    cuts = torch.tensor(np.cumsum(p / p.sum())[:-1], dtype=torch.float32, device="cuda")
    u = torch.rand(shape, generator=gen, device="cuda")
    w = torch.full(shape, lo, dtype=torch.int8, device="cuda")
    for k in range(len(v) - 1):
        w += u >= cuts[k]
    return w


def _scale_bias(w, a_bits, out_bits, res_scale=0.0):
    """The calibration of ``workloads.calibrated_scale_bias`` for unsigned activations, on the device."""
    mean, var = wl.code_moments(a_bits, api.UNSIGNED)
    f = w.reshape(w.shape[0], -1).float()
    scale = 1.0 / torch.sqrt(torch.clamp(var * (f * f).sum(1), min=1.0))
    bias = ((1 << out_bits) - 1) / 2.0 - mean * f.sum(1) * scale - res_scale * ((1 << out_bits) - 1) / 2.0
    return scale.contiguous(), bias.contiguous()


def _float_input(gen, shape, bits):
    return (torch.rand(shape, generator=gen, device="cuda") * (1 << bits) - 0.5) * ACT_SCALE


def _net_spec(case):
    if case["kind"] == "classifier":
        return wl.resnet18_full(case["batch"], case["hw"])
    spec = STACKS[case["stack"]](case["batch"], case["hw"])
    spec.a_bits, spec.w_bits = case["a_bits"], case["w_bits"]
    return spec


def _net_params(gen, spec):
    sign, params = wl.weight_sign(spec.w_bits), {}
    for layer in spec.layers:
        w = _zero_mean_weights(gen, (layer.O, layer.C, layer.k, layer.k), spec.w_bits, sign)
        scale, bias = _scale_bias(w, spec.a_bits, spec.a_bits, layer.res_scale if layer.res else 0.0)
        params[layer.name] = dict(w=w.cpu().numpy(), scale=scale.cpu().numpy(), bias=bias.cpu().numpy(), w_sign=sign)
    return params


def _conv_out(case):
    pad = case["k"] // 2
    return (case["H"] + 2 * pad - case["k"]) // case["stride"] + 1, (case["W"] + 2 * pad - case["k"]) // case["stride"] + 1


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "pack":
        shape = (case["N"], case["C"], case["H"], case["W"]) if case["layout"] == "nchw" else (case["N"], case["H"], case["W"], case["C"])
        x = _float_input(gen, shape, case["bits"]) if case["dtype"] == "f32" else _codes(gen, shape, case["bits"], api.UNSIGNED)
        return dict(case=case, x=x, layout=api.NCHW if case["layout"] == "nchw" else api.NHWC)
    if kind in ("net", "classifier"):
        spec = _net_spec(case)
        if kind == "classifier":
            params = _net_params(gen, spec.body)
            params["stem"] = dict(w=(torch.randn(64, 3, 7, 7, generator=gen, device="cuda") / math.sqrt(147.0)).cpu().numpy(),
                                  bias=(torch.randn(64, generator=gen, device="cuda") * 0.1).cpu().numpy())
            params["fc"] = dict(w=(torch.randn(spec.classes, 512, generator=gen, device="cuda") / math.sqrt(512.0)).cpu().numpy(),
                                bias=(torch.randn(spec.classes, generator=gen, device="cuda") * 0.1).cpu().numpy())
            images = torch.randn(case["batch"], 3, case["hw"], case["hw"], generator=gen, device="cuda")
            return dict(case=case, x=images, net=net.BitserialFullNet(spec, params, batch=case["batch"]))
        x = _float_input(gen, (case["batch"], *spec.in_shape), spec.a_bits)
        runner = net.BitserialNet(spec, _net_params(gen, spec), ACT_SCALE, batch=case["batch"], engine=case["engine"])
        if case["mode"] == "replay":
            runner.capture(x)
        return dict(case=case, x=x, net=runner)

    a, w = case["a_bits"], case["w_bits"]
    w_sign = wl.weight_sign(w)
    if kind == "gemm":
        rows = _codes(gen, (case["M"], case["K"]), a, api.UNSIGNED)
        filters = _codes(gen, (case["N"], case["K"]), w, w_sign)
        s = dict(case=case, a=api.bs_pack_rows(rows, a, api.UNSIGNED), w=api.bs_pack_rows(filters, w, w_sign), w_sign=w_sign)
        if case["engine"] == "tc" and api.tc_supported(1, case["K"], 1, case["M"], case["N"], 1, 1, 0, a, api.UNSIGNED, w, w_sign):
            s["w_tc"] = api.tc_prepare_weights(s["w"].view(case["N"], 1, 1, -1, w), case["K"], w_sign, a)
        s["kw"] = dict(a_sign=api.UNSIGNED, w_sign=w_sign)
        if case["out"] == "codes":
            s["scale"], s["bias"] = _scale_bias(filters, a, a)
            s["kw"].update(scale=s["scale"], bias=s["bias"], relu=True, out_bits=a, want_i32=False)
        return s

    pad = case["k"] // 2
    x = _codes(gen, (case["N"], case["C"], case["H"], case["W"]), a, api.UNSIGNED)
    filters = _zero_mean_weights(gen, (case["O"], case["C"], case["k"], case["k"]), w, w_sign)
    s = dict(case=case, a=api.bitpack_activations(x, 1.0, a), w=api.pack_weights(filters, w, w_sign))
    kw = dict(C=case["C"], stride=case["stride"], pad=pad, w_sign=w_sign)
    if case["engine"] == "tc" and api.tc_supported(case["N"], case["C"], case["H"], case["W"], case["O"], case["k"], case["stride"], pad,
                                                   a, api.UNSIGNED, w, w_sign):
        kw["wgt_tc"] = api.tc_prepare_weights(s["w"], case["C"], w_sign, a)
    if case["out"] == "acc":
        kw["want_i32"] = True
    else:
        res = wl.RES_SCALE if case["residual"] else 0.0
        scale, bias = _scale_bias(filters, a, a, res)
        kw.update(scale=scale, bias=bias, relu=True, out_bits=a)
        if case["residual"]:
            P, Q = _conv_out(case)
            codes = _codes(gen, (case["N"], case["O"], P, Q), a, api.UNSIGNED)
            kw.update(residual=api.bitpack_activations(codes, 1.0, a), res_scale=res, res_bits=a)
    s["kw"] = kw
    return s


# ----------------------------------------------------------------------------------------------------------- one pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "conv":
        acc, packed = api.bitserial_conv2d(state["a"], state["w"], **state["kw"])
        return acc if case["out"] == "acc" else packed
    if kind == "gemm":
        if "w_tc" in state:
            acc, packed = api.bitserial_gemm_tc(state["a"], state["w_tc"], case["N"], case["K"], case["w_bits"], **state["kw"])
        else:
            acc, packed = api.bitserial_gemm(state["a"], state["w"], case["K"], **state["kw"])
        return acc if case["out"] == "acc" else packed
    if kind == "pack":
        return api.bitpack_activations(state["x"], ACT_SCALE, case["bits"], api.UNSIGNED, state["layout"])
    if kind == "net" and case["mode"] == "replay":
        return state["net"].replay(state["x"])
    return state["net"].forward(state["x"])


def _words(c):
    return (c + 31) // 32


def work(case):
    kind = case["kind"]
    if kind == "conv":
        P, Q = _conv_out(case)
        a, w, O, C, k = case["a_bits"], case["w_bits"], case["O"], case["C"], case["k"]
        pixels = case["N"] * P * Q
        out = pixels * O * 4 if case["out"] == "acc" else pixels * _words(O) * a * 4 * (2 if case["residual"] else 1)
        read = case["N"] * case["H"] * case["W"] if k > 1 or case["stride"] == 1 else pixels
        return {"bytes": read * _words(C) * a * 4 + O * k * k * _words(C) * w * 4 + out, "flops": 2 * pixels * O * C * k * k}
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        out = M * N * 4 if case["out"] == "acc" else M * _words(N) * case["a_bits"] * 4
        return {"bytes": (M * case["a_bits"] + N * case["w_bits"]) * _words(K) * 4 + out, "flops": 2 * M * N * K}
    if kind == "pack":
        pixels = case["N"] * case["H"] * case["W"]
        values = pixels * case["C"]
        # a few comparisons for each value
        return {"bytes": values * (4 if case["dtype"] == "f32" else 1) + pixels * _words(case["C"]) * case["bits"] * 4, "flops": 4 * values}
    # a stack's tensors between its layers need not leave the chip: input, filters and the last codes (or the logits) have to move
    spec = _net_spec(case)
    body = spec.body if kind == "classifier" else spec
    filters = sum(L.O * L.k * L.k * _words(L.C) * body.w_bits * 4 for L in body.layers)
    if kind == "classifier":
        pixels = 3 * case["hw"] * case["hw"]
        return {"bytes": 4 * (case["batch"] * (pixels + spec.classes) + 64 * 147 + 512 * spec.classes) + filters,
                "flops": 2 * case["batch"] * (spec.stem_macs_per_image() + body.macs_per_image() + spec.head_macs_per_image())}
    C, H, W = spec.in_shape
    Co, P, Q = spec.tensor_shapes()[spec.out_name]
    return {"bytes": case["batch"] * (C * H * W * 4 + P * Q * _words(Co) * spec.a_bits * 4) + filters, "flops": 2 * case["batch"] * spec.macs_per_image()}


def tolerance(case):
    # codes and integer accumulators are exact; the logits are sums of 512 float32 products in a stated order
    return {"rel": 1e-5} if case["kind"] == "classifier" else "exact"
