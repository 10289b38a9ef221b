"""The work that users of this library have it do, as cases that can be timed and compared.

A case is a dict with a "kind" and sizes:

* conv, gemm -- one layer of a network at inference: the weights are ternarized once (groups of
  G, fp32 or fixed-point alphas), and each pass contracts a batch of quantized activations;
* latency    -- one layer at batch 1 with its activation quantizer, as an interactive user runs it;
* stem       -- the 8-bit-weight first layer of a network;
* ternarize  -- the weights of a whole network ternarized in one call (model preparation);
* quantize   -- the activations of a whole network quantized in one call (dynamic fixed point);
* forward    -- the chained ResNet forward at fixed scales (8-bit codes between the layers).

Sizes are those of the networks and sweeps in synth.py and bench.py; `draw` spreads over the same
ranges, ragged sizes among them.  Inputs follow synth.py's recipe: weights ~ N(0, 2 / fan_in),
activations half-normal (signed types: normal), drawn on the device from the seed.
"""
import math

import torch

from paper_1705_01462_gb300 import fgq, resnet, synth

QMAX = {"u8": 255, "s8": 127, "u4": 15, "s4": 7}
QMIN = {"u8": 0, "s8": -128, "u4": 0, "s4": -8}


def _conv(name, B, H, W, C, M, R, stride, pad, G, act="u8", groups=1, alpha="f32", out="f32"):
    return {"name": name, "kind": "conv", "B": B, "H": H, "W": W, "C": C, "M": M, "R": R, "S": R, "stride": stride,
            "pad": pad, "groups": groups, "G": G, "act": act, "alpha": alpha, "out": out}


def listed():
    return [
        # the smallest call: one image through the 3x3 layer of conv2_x, quantizer included
        dict(_conv("conv2x_3x3_b1_g4", 1, 56, 56, 64, 64, 3, 1, 1, 4), kind="latency"),
        # a fully connected layer for a single request: every weight read once
        {"name": "fc_4096_b1_g4", "kind": "gemm", "P": 1, "K": 4096, "M": 4096, "G": 4, "act": "u8", "alpha": "f32",
         "out": "f32"},
        # the bulk of a ResNet-50 at batch 64 and the paper's group size: a 3x3 layer of conv3_x
        _conv("res3_3x3_b64_g4", 64, 28, 28, 128, 128, 3, 1, 1, 4),
        # the coarser group size of the paper's accuracy comparison, a longer reduction
        _conv("res4_3x3_b64_g8", 64, 14, 14, 256, 256, 3, 1, 1, 8),
        # strided 1x1 projection at G = 64: little arithmetic, a large fp32 output
        _conv("res3_proj_b64_g64", 64, 56, 56, 256, 512, 1, 2, 0, 64),
        # 4-bit activations, G = 64, ResNet-101 at batch 128
        _conv("res4_3x3_b128_g64_u4", 128, 14, 14, 256, 256, 3, 1, 1, 64, act="u4"),
        # AlexNet's two-tower 5x5 layer: 48 channels per tower, signed activations; the most work
        _conv("alex_conv2_b256_g4_s8", 256, 27, 27, 96, 256, 5, 1, 2, 4, act="s8", groups=2),
        # a large fully connected layer at batch 256: weight-dominated
        {"name": "alex_fc6_b256_g4_s8", "kind": "gemm", "P": 256, "K": 9216, "M": 4096, "G": 4, "act": "s8",
         "alpha": "f32", "out": "f32"},
        # the first layer of a ResNet at batch 64, 8-bit weights
        {"name": "stem_b64_w8", "kind": "stem", "B": 64, "H": 224, "W": 224, "C": 3, "M": 64, "R": 7, "stride": 2,
         "pad": 3, "act": "u8"},
        # a network's weights ternarized when it is loaded: the last 31 convolutions, most of the weights
        {"name": "ternarize_resnet50_g4", "kind": "ternarize", "net": "resnet50", "first": 22, "count": 31, "G": 4},
        # the inputs of a network's layers quantized, each with its own scale: the first 31 convolutions
        {"name": "quantize_resnet50_b16", "kind": "quantize", "net": "resnet50", "first": 0, "count": 31, "B": 16,
         "act": "u8"},
        # a whole forward at fixed scales, codes between the layers
        {"name": "forward_resnet50_b16_g4", "kind": "forward", "B": 16, "hw": 224, "G": 4, "blocks": 16},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["conv", "gemm", "stem", "ternarize", "quantize", "forward", "latency"],
                       [10, 5, 2, 2, 2, 1, 1])[0]
    act = rng.choice(["u8", "u8", "s8", "u4", "s4"])
    G = rng.choice([4, 4, 8, 16, 32, 64, 64, 128])
    alpha = rng.choice(["f32", "f32", "f32", "a8", "a4"])
    out = rng.choice(["f32", "f32", "u8"]) if alpha == "f32" else "f32"
    if kind in ("conv", "latency"):
        while True:
            groups = rng.choice([1, 1, 1, 2])
            Cg = rng.choice([64, 128, 256, 512, 4 * rng.randint(8, 64), 16 * rng.randint(2, 32)])
            Mg = rng.choice([64, 128, 256, 512, 1024, rng.randint(16, 400)])
            R = rng.choice([1, 1, 3, 3, 5])
            H = rng.choice([7, 14, 28, 56, rng.randint(5, 60)])
            W = rng.choice([H, H, rng.randint(5, 60)])
            stride = rng.choice([1, 1, 1, 2])
            B = 1 if kind == "latency" else _logint(rng, 1, 128)
            Ho, Wo = (H + 2 * (R // 2) - R) // stride + 1, (W + 2 * (R // 2) - R) // stride + 1
            P, M = B * Ho * Wo, Mg * groups
            if 2 * M * P * R * R * Cg <= 4e10 and 4 * P * M <= 4e8 and B * H * W * Cg * groups <= 1e8:
                break
        c = _conv("", B, H, W, Cg * groups, M, R, stride, R // 2, G, act, groups, alpha, out)
        del c["name"]
        return dict(c, kind=kind) if kind == "conv" else dict(c, kind=kind, act="u8", alpha="f32", out="f32")
    if kind == "gemm":
        while True:
            P, K, M = _logint(rng, 1, 2048), 4 * _logint(rng, 64, 4096), _logint(rng, 100, 16384)
            if rng.random() < 0.6:
                K, M = (K + 63) // 64 * 64, (M + 3) // 4 * 4
            if 2.0 * P * K * M <= 6e10:
                return {"kind": kind, "P": P, "K": K, "M": M, "G": G, "act": act, "alpha": alpha, "out": out}
    if kind == "stem":
        R, stride, pad = rng.choice([(7, 2, 3), (11, 4, 0), (3, 1, 1)])
        H, W, M = rng.randint(60, 230), rng.randint(60, 230), rng.choice([32, 64, 96])
        B = min(_logint(rng, 1, 64), max(1, 10 ** 8 * stride * stride // (H * W * M)))
        return {"kind": kind, "B": B, "H": H, "W": W, "C": 3, "M": M, "R": R, "stride": stride, "pad": pad,
                "act": rng.choice(["u8", "s8"])}
    net = rng.choice(["resnet50", "resnet101", "alexnet"])
    n = len(_layers(net))
    count = rng.randint(1, min(n, 31))
    first = rng.randint(0, n - count)
    if kind == "ternarize":
        while sum(l.M * l.Kred for l in _layers(net)[first:first + count]) > 2.6e7:
            count //= 2
        return {"kind": kind, "net": net, "first": first, "count": count, "G": G}
    if kind == "quantize":
        B = _logint(rng, 1, 32)
        while sum(B * l.H * l.W * l.C for l in _layers(net)[first:first + count]) > 1.7e8 and count > 1:
            count //= 2
        return {"kind": kind, "net": net, "first": first, "count": count, "B": B, "act": act}
    return {"kind": "forward", "B": _logint(rng, 1, 16), "hw": 32 * rng.randint(2, 7), "G": rng.choice([4, 64]),
            "blocks": rng.choice([3, 7, 13, 16])}


def _layers(net):
    if net == "alexnet":
        return synth.alexnet_convs() + synth.alexnet_fcs()
    return synth.resnet101_convs() if net == "resnet101" else synth.resnet50_convs()


def _chain_layers(case):
    """conv1 and the first `blocks` bottleneck blocks of ResNet-50."""
    layers, blocks, keep = synth.resnet50_convs(), 0, []
    for l in layers:
        if l.name.endswith("branch2a"):
            blocks += 1
        if blocks > case["blocks"]:
            break
        keep.append(l)
    return keep


def _gen(seed, i=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * (int(seed) % 2000003) + 17 * i + 5)


def _normal(shape, seed, i):
    return torch.randn(shape, generator=_gen(seed, i), device="cuda", dtype=torch.float32)


# ------------------------------------------------------------- inputs (plain torch, no library code)

def _ternary(w, G):
    """Per group of G: the threshold maximising (sum of kept |w|)^2 / kept -> (t int8, alpha fp32)."""
    M, K = w.shape
    ng = (K + G - 1) // G
    g = torch.nn.functional.pad(w, (0, ng * G - K)).view(M, ng, G)
    a = g.abs().double()
    top = a.sort(dim=2, descending=True).values
    S = top.cumsum(2)
    k = torch.arange(1, G + 1, device=w.device, dtype=torch.float64)
    best = (S * S / k).argmax(2, keepdim=True)
    tau = top.gather(2, best)
    t = torch.where((a >= tau) & (a > 0), g.sign(), torch.zeros_like(g)).to(torch.int8)
    alpha = (S.gather(2, best) / (best + 1)).squeeze(2).float()
    return t.view(M, ng * G), alpha


def _pack_codes(t):
    M, Kp = t.shape
    wr = (Kp + 15) // 16
    c = torch.nn.functional.pad(t, (0, wr * 16 - Kp)).view(M, wr, 16).to(torch.int64) & 3
    w = (c << (2 * torch.arange(16, device=t.device))).sum(2)
    return torch.where(w >= 1 << 31, w - (1 << 32), w).to(torch.int32).contiguous()


def _dfp(x, qmax):
    m = x.abs().max().item()
    return 2.0 ** math.ceil(math.log2(m / qmax)) if m > 0 else 1.0


def _acts(shape, act, seed):
    x = _normal(shape, seed, 2)
    x = x.abs() if act[0] == "u" else x
    s = _dfp(x, QMAX[act])
    return torch.clamp(torch.round(x / s), QMIN[act], QMAX[act]).to(torch.int16), s


def _pack_acts(q, act):
    if act[1] == "8":
        return (q & 255).to(torch.uint8).contiguous()
    n = (q & 15).reshape(-1, 2)
    return (n[:, 0] | (n[:, 1] << 4)).to(torch.uint8).contiguous()


def _layer_inputs(case, seed):
    """Weights as (t, alpha, fixed-point alphas), activations as integers: kinds conv, latency, gemm."""
    M, G = case["M"], case["G"]
    K = case["K"] if case["kind"] == "gemm" else case["R"] * case["S"] * (case["C"] // case["groups"])
    t, alpha = _ternary(_normal((M, K), seed, 1) * math.sqrt(2.0 / K), G)
    aq = asc = None
    if case["alpha"] != "f32":  # 8- or 4-bit alphas, one power-of-two scale per filter
        top = 255.0 if case["alpha"] == "a8" else 15.0
        asc = torch.exp2(torch.ceil(torch.log2(alpha.max(1).values.double() / top)))
        aq = torch.clamp(torch.round(alpha.double() / asc[:, None]), 0, top)
    shape = (case["P"], K) if case["kind"] == "gemm" else (case["B"], case["H"], case["W"], case["C"])
    return t, alpha, aq, asc, shape


def _effective(case, t, alpha, aq, asc):
    """The weights alpha * t in fp64, [M][Kp]."""
    a = alpha.double() if aq is None else aq * asc[:, None]
    return t.double() * a.repeat_interleave(case["G"], dim=1)


def _out_scale(w, q, s):
    """A power of two that puts four standard deviations of the output at 127."""
    sd = s * math.sqrt(float((w * w).sum(1).mean()) * float(q.double().square().mean()))
    return 2.0 ** math.ceil(math.log2(4 * sd / 127))


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("conv", "gemm", "latency"):
        t, alpha, aq, asc, shape = _layer_inputs(case, seed)
        st["codes"], st["alpha"] = _pack_codes(t), alpha.contiguous()
        if kind == "latency":
            st["x"] = _normal(shape, seed, 2).abs()
            return st
        q, s = _acts(shape, case["act"], seed)
        st["q"] = _pack_acts(q, case["act"])
        st["scale"] = torch.tensor([s], dtype=torch.float32, device="cuda")
        if aq is not None:
            a = aq.to(torch.uint8)
            if case["alpha"] == "a4":
                a = torch.nn.functional.pad(a, (0, a.shape[1] % 2)).view(a.shape[0], -1, 2)
                a = a[:, :, 0] | (a[:, :, 1] << 4)
            st["aq"], st["ascale"] = a.contiguous(), asc.float()
        if case["out"] == "u8":
            o = _out_scale(_effective(case, t, alpha, aq, asc), q, s)
            st["oscale"] = torch.tensor([o], dtype=torch.float32, device="cuda")
    elif kind == "stem":
        wq, ws, q, s = _stem_inputs(case, seed)
        st["wq"], st["wscale"] = wq.to(torch.int8), ws.float()
        st["q"] = _pack_acts(q, case["act"])
        st["scale"] = torch.tensor([s], dtype=torch.float32, device="cuda")
    elif kind == "ternarize":
        st["w"] = [_normal((l.M, l.Kred), seed, 100 + i) * math.sqrt(2.0 / l.fan_in)
                   for i, l in enumerate(_layers(case["net"])[case["first"]:case["first"] + case["count"]])]
    elif kind == "quantize":
        st["x"] = []
        for i, l in enumerate(_layers(case["net"])[case["first"]:case["first"] + case["count"]]):
            x = _normal((case["B"], l.H, l.W, l.C), seed, 100 + i)
            st["x"].append(x.abs() if case["act"][0] == "u" else x)
    else:
        # weights in {-c, 0, +c} with c a power of two are ternary already and every sum is exact in
        # fp32, so that a chain of 50 layers gives the same codes in any order of summation (with
        # other weights a rounding difference at a code boundary spreads from layer to layer)
        layers = _chain_layers(case)
        params, dev = [], torch.device("cuda")
        for i, l in enumerate(layers):
            w = _normal((l.M, l.Kred), seed, 100 + i)
            c = 2.0 ** round(math.log2(math.sqrt(3.0 / l.fan_in)))
            if i > 0:
                w = torch.where(w.abs() > 0.6, c * w.sign(), torch.zeros_like(w))
                params.append(fgq.fgq_ternarize(w, case["G"]))
            else:
                params.append(None)
                w8 = fgq.fgq_quantize_weights_w8(w * math.sqrt(2.0 / l.fan_in))
        st["net"] = resnet.QuantResNet(layers, case["G"], dev, params=(w8, params))
        st["x"] = _normal((case["B"], case["hw"], case["hw"], 3), seed, 2).abs()
        st["net"].calibrate(st["x"])
    return st


def _stem_inputs(case, seed):
    K = case["R"] * case["R"] * case["C"]
    w = (_normal((case["M"], K), seed, 1) * math.sqrt(2.0 / K)).double()
    ws = torch.exp2(torch.ceil(torch.log2(w.abs().max(1).values / 127.0)))
    wq = torch.clamp(torch.round(w / ws[:, None]), -128, 127)
    q, s = _acts((case["B"], case["H"], case["W"], case["C"]), case["act"], seed)
    return wq, ws, q, s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ternarize":
        return fgq.fgq_ternarize_batch(state["w"], case["G"])
    if kind == "quantize":
        return fgq.fgq_quantize_act_batch(state["x"], [case["act"]] * len(state["x"]))
    if kind == "forward":
        y = state["net"].forward_fused(state["x"])
        return [y.q, y.scale]
    if kind == "stem":
        return fgq.fgq_conv2d_w8(state["q"], case["act"], state["scale"], case["B"], case["H"], case["W"], case["C"],
                                 case["R"], case["R"], case["stride"], case["pad"], 1, state["wq"], state["wscale"],
                                 case["M"])
    if kind == "gemm":
        geo = (case["P"], case["K"])
        f32, rq, qa = fgq.fgq_gemm, fgq.fgq_gemm_rq, fgq.fgq_gemm_qa
    else:
        geo = tuple(case[k] for k in ("B", "H", "W", "C", "R", "S", "stride", "pad", "groups"))
        f32, rq, qa = fgq.fgq_conv2d, fgq.fgq_conv2d_rq, fgq.fgq_conv2d_qa
    if kind == "latency":
        q, s = fgq.fgq_quantize_act(state["x"], case["act"])
        return [q, s, f32(q, case["act"], s, *geo, state["codes"], state["alpha"], case["M"], case["G"])]
    head = (state["q"], case["act"], state["scale"]) + geo + (state["codes"],)
    if case["alpha"] != "f32":
        return qa(*head, state["aq"], 8 if case["alpha"] == "a8" else 4, state["ascale"], case["M"], case["G"])
    if case["out"] == "u8":
        return rq(*head, state["alpha"], case["M"], case["G"], "u8", state["oscale"])
    return f32(*head, state["alpha"], case["M"], case["G"])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("conv", "gemm", "latency"):
        t, alpha, aq, asc, shape = _layer_inputs(case, seed)
        if case["out"] != "f32":
            return None
        if kind == "latency":
            x = _normal(shape, seed, 2).abs()
            s = _dfp(x, QMAX[case["act"]])
            q = torch.clamp(torch.round(x / s), QMIN[case["act"]], QMAX[case["act"]])
        else:
            q, s = _acts(shape, case["act"], seed)
        w = _effective(case, t, alpha, aq, asc)
        if kind == "gemm":
            return s * (q.double() @ w[:, :case["K"]].t())
        y = s * _conv64(q.double(), w, case["R"], case["S"], case["stride"], case["pad"], case["groups"])
        return [None, torch.tensor([s], dtype=torch.float64), y] if kind == "latency" else y
    if kind == "stem":
        wq, ws, q, s = _stem_inputs(case, seed)
        return s * _conv64(q.double(), wq * ws[:, None], case["R"], case["R"], case["stride"], case["pad"], 1)
    return None  # whole numbers, compared bit for bit


def _conv64(x, w, R, S, stride, pad, groups):
    """NHWC convolution in fp64, one tap at a time; w [M][>= R S C / groups] in (r, s, c) order."""
    B, H, W, C = x.shape
    M, Cg = w.shape[0], C // groups
    Ho, Wo = (H + 2 * pad - R) // stride + 1, (W + 2 * pad - S) // stride + 1
    x = torch.nn.functional.pad(x, (0, 0, pad, pad, pad, pad))
    y = torch.zeros((B, Ho, Wo, M), dtype=torch.float64, device=x.device)
    for g in range(groups):
        ms, cs = slice(g * M // groups, (g + 1) * M // groups), slice(g * Cg, (g + 1) * Cg)
        for r in range(R):
            for s in range(S):
                k = (r * S + s) * Cg
                xt = x[:, r:r + (Ho - 1) * stride + 1:stride, s:s + (Wo - 1) * stride + 1:stride, cs]
                y[..., ms] += xt @ w[ms, k:k + Cg].t()
    return y


def work(case):
    kind = case["kind"]
    if kind == "ternarize":
        ls = _layers(case["net"])[case["first"]:case["first"] + case["count"]]
        n, g = sum(l.M * l.Kred for l in ls), sum(l.M * -(-l.Kred // case["G"]) for l in ls)
        return {"bytes": 4 * n + n / 4 + 4 * g, "flops": 0}
    if kind == "quantize":
        n = sum(case["B"] * l.H * l.W * l.C for l in _layers(case["net"])[case["first"]:case["first"] + case["count"]])
        return {"bytes": n * (4 + int(case["act"][1]) / 8), "flops": 0}
    if kind == "forward":
        by, fl, B, f = 4.0 * case["B"] * case["hw"] ** 2 * 3, 0.0, case["B"], (case["hw"] / 224.0) ** 2
        for i, l in enumerate(_chain_layers(case)):  # codes in and out of every layer
            by += f * B * (l.H * l.W * l.C + l.Ho * l.Wo * l.M) + l.M * l.Kred * (1 if i == 0 else 0.25 + 4 / case["G"])
            fl += f * l.ops(B)
        return {"bytes": by, "flops": fl}
    if kind == "gemm":
        P, K, n, M = case["P"], case["K"], case["P"] * case["K"], case["M"]
    else:
        S = case.get("S", case["R"])
        Ho = (case["H"] + 2 * case["pad"] - case["R"]) // case["stride"] + 1
        Wo = (case["W"] + 2 * case["pad"] - S) // case["stride"] + 1
        P, M = case["B"] * Ho * Wo, case["M"]
        K = case["R"] * S * case["C"] // case.get("groups", 1)
        n = case["B"] * case["C"] * (Ho * Wo if case["R"] == 1 and case["pad"] == 0 else case["H"] * case["W"])
    flops = 2.0 * M * P * K
    if kind == "stem":
        return {"bytes": n + M * K + 4 * M + 4 * P * M, "flops": flops}
    ab = {"f32": 4, "a8": 1, "a4": 0.5}[case["alpha"]]
    acts = n * 5 if kind == "latency" else n * int(case["act"][1]) / 8
    return {"bytes": acts + M * K / 4 + ab * M * -(-K // case["G"]) + P * M * (4 if case["out"] == "f32" else 1),
            "flops": flops}


def tolerance(case):
    if case["kind"] in ("conv", "gemm", "latency") and case["alpha"] == "f32":
        # fp32 sums of alpha * (exact integers): relative to the output's norm, and per element to its
        # root mean square; requantized codes may differ where the sum lies at a rounding boundary
        return {"rel": 1.5e-6, "max": 1.5e-5, "differ": 0.0 if case["out"] == "f32" else 5e-4}
    if case["kind"] in ("conv", "gemm"):
        # fixed-point alphas: integer sums, rounded once where they stay below 2^24
        return {"rel": 1.5e-6, "max": 1.5e-5}
    if case["kind"] == "stem":
        return {"rel": 1e-6, "max": 1e-5}
    return "exact"
