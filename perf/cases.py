"""Performance cases: the work a user of the library has it do.

Each case is one call (or one network forward) through the public Python
entry points, on inputs of the library's own workloads: the LeNet-like layer,
the convolutions of the VGG-small, AlexNet and ResNet-18 shaped networks,
their backward products, the fully-connected sizes of the GEMV sweep, the
quantizer, and whole networks.  ``listed`` names the fixed ones, ``draw``
gives more of the same ranges, ``exact`` the same results in 64 bits from
plain torch.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

import paper_1701_00485_gb300 as tbn
from paper_1701_00485_gb300 import inputs, nets

DEV = "cuda"


# ------------------------------------------------------------------ cases
def _conv(name, kind, N, C, H, W, K, R, stride, pad, **more):
    c = dict(name=name, kind=kind, N=N, C=C, H=H, W=W, K=K, R=R, S=R, stride=stride, pad=pad)
    c.update(more)
    return c


def listed():
    return [
        # the LeNet-like layer: fp32 NCHW, quantized and convolved in every
        # step; the smallest work, where launches and the host path count
        _conv("lenet_quant_conv_b16", "quant_conv", 16, 1, 28, 28, 20, 5, 1, 0, f32=True),
        # one image through a middle ResNet-18 layer with its shortcut:
        # single-request inference
        _conv("conv_256_14x14_b1", "conv", 1, 256, 14, 14, 256, 3, 1, 1, relu=True, residual=True,
              pool=0, out_f32=False),
        # VGG-small's fourth layer at its batch, ReLU and 2x2 pool fused
        _conv("conv_256_16x16_b128_pool", "conv", 128, 256, 16, 16, 256, 3, 1, 1, relu=True,
              residual=False, pool=2, out_f32=False),
        # a first-stage ResNet-18 layer (64 filters, few channels, large maps)
        _conv("conv_64_56x56_b64_residual", "conv", 64, 64, 56, 56, 64, 3, 1, 1, relu=True,
              residual=True, pool=0, out_f32=False),
        # a channel count that is no multiple of 32, odd maps, fp32 output
        _conv("conv_40_27x27_b32_odd", "conv", 32, 40, 27, 27, 128, 5, 1, 2, relu=False,
              residual=False, pool=0, out_f32=True),
        # training: both gradients of VGG-small's third layer
        _conv("backward_128_256_16x16_b128", "backward", 128, 128, 16, 16, 256, 3, 1, 1),
        # the largest batch-1 layer of the GEMV sweep
        dict(name="linear_16384_b1", kind="linear", B=1, K_in=16384, K_out=16384, f32=False),
        # its smallest size at batch 8
        dict(name="linear_4096_b8", kind="linear", B=8, K_in=4096, K_out=4096, f32=False),
        # fp32 activations at batch 1
        dict(name="linear_8192_b1_f32", kind="linear", B=1, K_in=8192, K_out=8192, f32=True),
        # the quantizer on a large layer
        dict(name="quantize_8192x8192", kind="quantize", K=8192, n=8192),
        # whole networks: AlexNet re-quantized in each step (Algorithm 1), and
        # ResNet-18 in its inference form
        dict(name="alexnet_b256", kind="net", net="alexnet", N=256, requantize=True),
        dict(name="resnet18_b128", kind="net", net="resnet18", N=128, requantize=False),
    ]


def _log(rng, lo, hi):
    """An integer of [lo, hi], uniform over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _channels(rng, hi):
    """Channel counts: mostly the multiples of 64 that networks have, also of
    32 and 8, sometimes any number."""
    step = rng.choice((64, 64, 64, 32, 8, 1))
    return max(step, _log(rng, min(step, 16), hi) // step * step)


def draw(rng):
    kind = rng.choice(("quant_conv", "conv", "conv", "conv", "backward", "linear", "linear",
                       "quantize", "net"))
    if kind == "quantize":
        K, n = _log(rng, 16, 8192), _log(rng, 25, 8192)
        return dict(kind=kind, K=K, n=n)
    if kind == "linear":
        f32 = rng.random() < 0.25
        B = 1 if f32 else rng.choice((1, 1, 2, 3, 5, 8, 8, 16, 64, 100, 256))
        step = 64 if f32 else rng.choice((64, 64, 8))
        K_in = max(step, _log(rng, 256, 16384) // step * step)
        return dict(kind=kind, B=B, K_in=K_in, K_out=_log(rng, 10, 16384), f32=f32)
    if kind == "net":
        net = rng.choice(("vgg_small", "alexnet", "resnet18"))
        most = dict(vgg_small=128, alexnet=256, resnet18=128)[net]
        # smaller steps than the listed networks: their batch is the largest
        return dict(kind=kind, net=net, N=_log(rng, 1, most - 1),
                    requantize=net != "resnet18" and rng.random() < 0.5)
    if kind == "quant_conv":
        # small fp32 layers in NCHW, as LeNet's
        while True:
            R = rng.choice((3, 5))
            c = _conv(None, kind, _log(rng, 1, 64), rng.choice((1, 3, 6, 16, 20)),
                      rng.randint(7, 32), rng.randint(7, 32), rng.randint(6, 64), R, 1,
                      rng.choice((0, R // 2)), f32=True)
            if _conv_flops(c) <= 3e8:
                break
    else:
        while True:
            R = rng.choice((1, 3, 3, 3, 5))
            H = _log(rng, 7, 56)
            c = _conv(None, kind, _log(rng, 1, 128), _channels(rng, 512), H,
                      max(7, H + rng.choice((0, 0, 0, 1, -1, 4))), _channels(rng, 512), R,
                      rng.choice((1, 1, 1, 2)), R // 2)
            if (1e6 <= _conv_flops(c) <= (4e10 if c["C"] % 32 == 0 else 1e10) and
                    c["N"] * c["H"] * c["W"] * max(c["C"], c["K"]) <= 3e7):
                break
        if kind == "backward":
            c["C"], c["K"] = max(8, c["C"] // 8 * 8), max(8, c["K"] // 8 * 8)
        else:
            glue = rng.choice(("none", "relu", "residual", "pool"))
            P, Q = _out_hw(c)
            if glue == "pool" and (P < 2 or Q < 2):
                glue = "relu"
            c.update(relu=glue != "none", residual=glue == "residual",
                     pool=2 if glue == "pool" else 0, out_f32=rng.random() < 0.2)
    del c["name"]
    return c


# ------------------------------------------------------------------ sizes
def _out_hw(c):
    return tuple((d + 2 * c["pad"] - r) // c["stride"] + 1
                 for d, r in ((c["H"], c["R"]), (c["W"], c["S"])))


def _conv_flops(c):
    P, Q = _out_hw(c)
    return 2.0 * c["N"] * c["K"] * P * Q * c["C"] * c["R"] * c["S"]


def _code_bytes(K, n):
    return 4.0 * K * ((n + 15) // 16) + 4.0 * K


def _net_layers(c):
    """(K, n, outputs per filter, two-bit) of every layer with weights."""
    N = c["N"]
    if c["net"] == "resnet18":
        hw = {"l1": 56, "l2": 28, "l3": 14, "l4": 7}
        out = [(64, 147, N * 112 * 112, False)]
        out += [(s.K, s.C * s.R * s.S, N * hw[name[:2]] ** 2, True)
                for name, s in inputs.resnet18_convs()]
        return out + [(1000, 512, N, False)]
    cfg = inputs.ALEXNET if c["net"] == "alexnet" else inputs.VGG_SMALL
    h, out = cfg["H"], []
    for s in cfg["convs"]:
        h = (h + 2 * s.pad - s.R) // s.stride + 1
        out.append((s.K, s.C * s.R * s.S, N * h * h, True))
        if s.pool:
            h = (h - s.pool[0]) // s.pool[1] + 1
    return out + [(o, i, N, True) for i, o, _ in cfg.get("fcs", [])]


def work(case):
    k = case["kind"]
    if k == "quantize":
        n = case["K"] * case["n"]
        return {"bytes": 4.0 * n + _code_bytes(case["K"], case["n"]), "flops": 2.0 * n}
    if k == "linear":
        B, i, o = case["B"], case["K_in"], case["K_out"]
        e = 4 if case["f32"] else 2
        return {"bytes": _code_bytes(o, i) + e * B * (i + o), "flops": 2.0 * B * i * o}
    if k == "net":
        hw = {"vgg_small": 32, "alexnet": 227, "resnet18": 224}[case["net"]]
        layers = _net_layers(case)
        b = 2.0 * case["N"] * 3 * hw * hw
        for K, n, _, two in layers:
            b += 4.0 * K * n if case["requantize"] or not two else 0.0
            b += _code_bytes(K, n) if two else 0.0
        b += (4.0 if case["net"] == "resnet18" else 2.0) * layers[-1][0] * layers[-1][2] / (
            4 if case["net"] == "vgg_small" else 1)      # the last map is pooled 2x2
        return {"bytes": b, "flops": sum(2.0 * K * n * m for K, n, m, _ in layers)}
    n = case["C"] * case["R"] * case["S"]
    P, Q = _out_hw(case)
    x = float(case["N"] * case["C"] * case["H"] * case["W"])
    y = float(case["N"] * case["K"] * P * Q)
    codes = _code_bytes(case["K"], n)
    if k == "quant_conv":
        return {"bytes": 4.0 * (case["K"] * n + x + y) + codes, "flops": _conv_flops(case)}
    if k == "backward":   # reads x, dy and the codes, writes dx (bf16) and dW (fp32)
        return {"bytes": 2.0 * (2 * x + y) + codes + 4.0 * case["K"] * n,
                "flops": 2 * _conv_flops(case)}
    if case["pool"]:
        y = float(case["N"] * case["K"] * (P // 2) * (Q // 2))
    e = 4.0 if case["out_f32"] else 2.0
    return {"bytes": 2.0 * x + codes + e * y * (2 if case["residual"] else 1),
            "flops": _conv_flops(case)}


def tolerance(case):
    """About four times what the path shows against ``exact``."""
    k = case["kind"]
    if k == "quantize":       # codes bit for bit; alpha is one rounding of an exact sum
        return {"rel": 2e-7, "max": 6e-7, "differ": 0.0}
    if k == "quant_conv":     # fp32 sums of at most 500 terms
        return {"rel": 1.5e-6, "max": 1e-5, "differ": 0.0}
    if k == "backward":       # dx: alpha * dy and dx rounded to bf16; dW: fp32 sums
        return {"rel": 9e-3, "max": 7e-2}
    if k == "net":            # every layer's output is rounded to bf16
        rel = {"vgg_small": 1.4e-2, "alexnet": 1.8e-2, "resnet18": 3.6e-3}[case["net"]]
        return {"rel": rel, "max": 5 * rel, "differ": 0.0}
    if case.get("out_f32") or case.get("f32"):    # fp32 sums of up to 16384 terms
        return {"rel": 1.4e-6, "max": 8e-6}
    return {"rel": 7e-3, "max": 1.6e-2}           # one bf16 rounding of the output


# ----------------------------------------------------------------- states
def _randn(g, *shape, std=1.0, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32).mul_(std).to(dtype)


def _layer_data(case, seed):
    """x (and the other activations) and the fp32 filters of a single layer."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    k = case["kind"]
    if k == "quantize":
        # trained filters reach past the threshold |W| = 1 now and then
        return {"W": _randn(g, case["K"], case["n"], std=0.6)}
    if k == "linear":
        dt = torch.float32 if case["f32"] else torch.bfloat16
        return {"x": _randn(g, case["B"], case["K_in"], dtype=dt),
                "W": _randn(g, case["K_out"], case["K_in"], std=math.sqrt(2.0 / case["K_in"]))}
    N, C, H, W, K, R, S = (case[i] for i in ("N", "C", "H", "W", "K", "R", "S"))
    P, Q = _out_hw(case)
    if k == "quant_conv":
        return {"x": torch.rand(N, C, H, W, generator=g, device=DEV),
                "W": _randn(g, K, C * R * S, std=0.1)}
    d = {"x": _randn(g, N, H, W, C, dtype=torch.bfloat16),
         "W": _randn(g, K, R * S * C, std=math.sqrt(2.0 / (C * R * S)))}
    if k == "backward":
        d["dy"] = _randn(g, N, P, Q, K, dtype=torch.bfloat16)
    elif case["residual"]:
        d["residual"] = _randn(g, N, P, Q, K,
                               dtype=torch.float32 if case["out_f32"] else torch.bfloat16)
    return d


def prepare(case, seed):
    k = case["kind"]
    if k == "net":
        net = getattr(nets, case["net"])(batch=case["N"], seed=seed)
        net.quantize()        # the inference form keeps only codes and alpha
        return {"case": case, "net": net}
    d = _layer_data(case, seed)
    d["case"] = case
    if k in ("conv", "backward", "linear"):
        d["codes"], d["alpha"] = tbn.tbn_quantize_pack(d.pop("W"))
    if k == "linear":
        n = tbn.tbn_linear_workspace_bytes(case["B"], case["K_in"], case["K_out"], d["x"].dtype)
        d["workspace"] = torch.empty(n, dtype=torch.uint8, device=DEV) if n else None
    return d


def run(state):
    c = state["case"]
    k = c["kind"]
    if k == "quantize":
        return tbn.tbn_quantize_pack(state["W"])
    if k == "linear":
        return tbn.tbn_linear_fwd_ws(state["x"], state["codes"], state["alpha"], c["K_out"],
                                     state["workspace"])
    if k == "net":
        net = state["net"]
        y = net.forward(requantize=c["requantize"])
        if not c["requantize"]:
            return {"y": y}
        return {"y": y, "codes": [q[1] for q in _jobs(net)], "alpha": [q[2] for q in _jobs(net)]}
    geo = dict(stride=(c["stride"],) * 2, pad=(c["pad"],) * 2)
    if k == "quant_conv":
        codes, alpha = tbn.tbn_quantize_pack(state["W"])
        y = tbn.tbn_conv2d_fwd(state["x"], codes, alpha, c["K"], c["R"], c["S"],
                               layout=tbn.TBN_NCHW, **geo)
        return {"y": y, "codes": codes, "alpha": alpha}
    if k == "backward":
        dx = tbn.tbn_conv2d_bwd_data(state["dy"], state["codes"], state["alpha"], c["C"],
                                     (c["H"], c["W"]), c["R"], c["S"], **geo)
        dw = tbn.tbn_conv2d_bwd_filter(state["x"], state["dy"], c["R"], c["S"], **geo)
        return {"dx": dx, "dw": dw}
    return tbn.tbn_conv2d_fwd(state["x"], state["codes"], state["alpha"], c["K"], c["R"], c["S"],
                              layout=tbn.TBN_NHWC, relu=c["relu"], pool=c["pool"],
                              residual=state.get("residual"),
                              out_dtype=torch.float32 if c["out_f32"] else torch.bfloat16, **geo)


def _jobs(net):
    """(W, codes, alpha) of every two-bit layer of a chain network."""
    convs = net.features.layers if isinstance(net, nets.AlexNet) else net.layers
    jobs = [(l.W, l.codes, l.alpha) for l in convs]
    if isinstance(net, nets.AlexNet):
        jobs += [(l[0], l[1], l[2]) for l in net.classifier.layers]
    return jobs


# ------------------------------------------------------- results in 64 bits
def _two_bit(W):
    """alpha [K] and alpha * W~ [K, n] of fp32 filters, in 64 bits (Eq. 3 and 5)."""
    a = W.double().abs()
    two = a > 1
    alpha = (a * (1 + two.double())).sum(1) / (W.shape[1] + 3 * two.sum(1)).double()
    wt = torch.where(W > 0, 1.0, -1.0).double() * (1 + two.double())
    return alpha, alpha[:, None] * wt


def _conv64(x, w, stride, pad):
    """fp64 convolution of NCHW x in groups of images (bounded memory)."""
    step = max(1, int(2e8 // (w.shape[1] * w.shape[2] * w.shape[3] *
                              x.shape[2] * x.shape[3] / (stride * stride))))
    return torch.cat([F.conv2d(x[i:i + step].double(), w, stride=stride, padding=pad)
                      for i in range(0, x.shape[0], step)])


def _kcrs(W, K, C, R, S):
    return W.reshape(K, R, S, C).permute(0, 3, 1, 2).contiguous()


def _net64(case, seed):
    two = lambda W: _two_bit(W.to(DEV).reshape(W.shape[0], -1))   # noqa: E731
    if case["net"] == "resnet18":
        x, stem, convs, fc = inputs.resnet18_inputs(seed, case["N"])
        h = F.max_pool2d(_conv64(x.to(DEV), stem.to(DEV).double(), 2, 3).relu(), 3, 2, 1)
        ws = {name: (s, two(W)[1].reshape(W.shape)) for name, s, W in convs}
        conv = lambda name, v: _conv64(v, ws[name][1], ws[name][0].stride,   # noqa: E731
                                       ws[name][0].pad)
        for name, _, _ in convs:
            if name[-1] != "a":
                continue
            blk = name[:4]
            y = conv(blk + "b", conv(blk + "a", h).relu())
            h = (y + (conv(blk + "d", h) if blk + "d" in ws else h)).relu()
        return {"y": h.mean((2, 3)) @ fc.to(DEV).double().t()}
    alex = case["net"] == "alexnet"
    cfg = inputs.ALEXNET if alex else inputs.VGG_SMALL
    got = (inputs.alexnet_inputs if alex else inputs.vgg_small_inputs)(seed, case["N"])
    h, alphas = got[0].to(DEV), []
    for s, W in zip(cfg["convs"], got[1]):
        alpha, w = two(W)
        alphas.append(alpha)
        h = _conv64(h, w.reshape(W.shape), s.stride, s.pad).relu()
        if s.pool:
            h = F.max_pool2d(h, *s.pool)
    h = h.permute(0, 2, 3, 1)
    if alex:
        h = h.reshape(case["N"], -1)
        for (_, _, relu), W in zip(cfg["fcs"], got[2]):
            alpha, w = two(W)
            alphas.append(alpha)
            h = h @ w.t()
            h = h.relu() if relu else h
    out = {"y": h}
    if case["requantize"]:
        out.update(codes=[None] * len(alphas), alpha=alphas)
    return out


def exact(case, seed):
    k = case["kind"]
    if k == "net":
        return _net64(case, seed)
    d = _layer_data(case, seed)
    if k == "quantize":
        step = 1024
        alpha = torch.cat([_two_bit(d["W"][i:i + step])[0] for i in range(0, case["K"], step)])
        return (None, alpha)
    alpha, w = _two_bit(d["W"])
    if k == "linear":
        return d["x"].double() @ w.t()
    K, C, R, S = (case[i] for i in ("K", "C", "R", "S"))
    if k == "quant_conv":
        y = _conv64(d["x"], w.reshape(K, C, R, S), case["stride"], case["pad"])
        return {"y": y, "codes": None, "alpha": alpha}
    w = _kcrs(w, K, C, R, S)
    x = d["x"].permute(0, 3, 1, 2)
    if k == "backward":
        return _backward64(case, x, d["dy"].permute(0, 3, 1, 2), w)
    y = _conv64(x, w, case["stride"], case["pad"]).permute(0, 2, 3, 1)
    if case["residual"]:
        y = y + d["residual"].double()
    y = y.relu() if case["relu"] else y
    if case["pool"]:
        y = F.max_pool2d(y.permute(0, 3, 1, 2), 2, 2).permute(0, 2, 3, 1)
    return y.contiguous()


def _backward64(case, x, dy, w):
    """dx (NHWC) and dW ([K, R*S*C]) by one fp64 matrix product per tap."""
    K, C, R, S = w.shape
    st, p = case["stride"], case["pad"]
    P, Q = _out_hw(case)
    g = dy.permute(1, 0, 2, 3).reshape(K, -1).double()
    xp = F.pad(x.double(), (p, p, p, p))
    dxp, dw = torch.zeros_like(xp), torch.empty(K, R, S, C, dtype=torch.float64, device=DEV)
    for r in range(R):
        for s in range(S):
            at = (slice(None), slice(None), slice(r, r + st * (P - 1) + 1, st),
                  slice(s, s + st * (Q - 1) + 1, st))
            dw[:, r, s] = g @ xp[at].permute(0, 2, 3, 1).reshape(-1, C)
            dxp[at] += (w[:, :, r, s].t() @ g).reshape(C, -1, P, Q).permute(1, 0, 2, 3)
    dx = dxp[:, :, p:p + case["H"], p:p + case["W"]]
    return {"dx": dx.permute(0, 2, 3, 1).contiguous(), "dw": dw.reshape(K, -1)}
