"""The work a training program asks of this library, as measurable cases.

A case is one call (or the short run of calls that belong together) of the public entry
points on seeded synthetic tensors: whole layer steps at 4, 6 and 8 bits, the quantizer, the
fully-quantized L1 batch normalization, packed storage of saved codes, and a chain of two
layers.  `listed()` holds the shapes of the repository's own workloads and tests,
`draw()` further ones of the same ranges, ragged sizes among them.
"""
from __future__ import annotations

import math

import torch

from paper_2411_10948_gb300 import layer as L
from paper_2411_10948_gb300 import native as N

GROUPS = 4
SEED = 0x5EED


def listed():
    return [
        # A small layer on a short batch: 256 tokens, 512 -> 512.  Every kernel of the step
        # takes a few microseconds, so launches and their gaps are what it costs.
        dict(name="layer_small", kind="layer", mode="call", M=256, K=512, N=512, bits=4,
             x="channels", g="normal", sigma=1.5),
        # A ResNet 3x3 convolution 256 -> 256 as im2col GEMMs (batch 64, 14 x 14): wide
        # activation, narrow gradient, 4-bit codes.
        dict(name="layer_conv3x3", kind="layer", mode="call", M=12544, K=2304, N=256, bits=4,
             x="relu", g="normal", sigma=2.0),
        # The first linear layer of a ViT-B MLP at 64 x 197 tokens: the ordinary transformer
        # layer, 6-bit codes.
        dict(name="layer_vit_fc1", kind="layer", mode="call", M=12608, K=768, N=3072, bits=6,
             x="outlier", g="laplace", sigma=2.0),
        # The up projection of a large MLP, the largest layer, replayed from a CUDA graph with
        # its quantizer chains on three streams as a training loop runs it.
        dict(name="layer_large_up", kind="layer", mode="graph", M=16384, K=4096, N=11008, bits=6,
             x="outlier", g="laplace", sigma=2.5),
        # The down projection at 8 bits on a shorter batch: K loops of many exact chunks.
        dict(name="layer_large_down_8bit", kind="layer", mode="call", M=4096, K=11008, N=4096,
             bits=8, x="outlier", g="laplace", sigma=2.5),
        # Odd sizes everywhere: rows of neither input nor output are 16-byte aligned, as with
        # the last partial batch of an epoch and a head of an odd number of classes.
        dict(name="layer_ragged", kind="layer", mode="call", M=5003, K=1155, N=1001, bits=6,
             x="outlier", g="laplace", sigma=2.0),
        # An 8-bit layer whose inner indices run in group order (no folded shifts).
        dict(name="layer_grouped_8bit", kind="layer", mode="grouped", M=12608, K=768, N=3072,
             bits=8, x="outlier", g="laplace", sigma=2.0),
        # The gradient of a 7x7x3 stem convolution's im2col matrix (147 columns): a long,
        # narrow, unaligned tensor quantized alone, stochastic rounding, codes and transpose.
        dict(name="quantize_stem", kind="quantize", M=100352, C=147, bits=4, stochastic=True,
             transposed=True, x="laplace", sigma=2.0),
        # Batch normalization after an early convolution (56 x 56 x 64, batch 64), both
        # directions.
        dict(name="l1bn_early", kind="l1bn", R=200704, C=64, bits=8),
        # ... and after a bottleneck's last convolution (7 x 7 x 2048, batch 64).
        dict(name="l1bn_wide", kind="l1bn", R=3136, C=2048, bits=8),
        # The activation codes of the convolution above, packed for the backward pass and
        # expanded again.
        dict(name="pack_saved", kind="pack", M=12544, C=2304, bits=4),
        # A whole MLP, forward through both layers and then backward, the range passes of the
        # inner tensors formed by the GEMMs that write them.
        dict(name="chain_vit_mlp", kind="chain", M=12608, K=768, H=3072, N=768, bits=6),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """A size of the range, over its logarithm: as it falls (mostly odd sizes), or rounded to
    a multiple of 4 or of 64 as layers usually have it."""
    n = _log_uniform(rng, lo, hi)
    step = rng.choice((1, 4, 64, 64))
    return max(lo, min(hi, (n + step // 2) // step * step))


def draw(rng):
    kind = rng.choice(("layer", "layer", "layer", "quantize", "l1bn", "pack", "chain"))
    if kind == "layer":
        mode = rng.choice(("call", "call", "graph", "grouped"))
        while True:
            M, K, Nn = _size(rng, 64, 16384), _size(rng, 64, 11008), _size(rng, 64, 11008)
            if M * K * Nn <= 16384 * 4096 * 11008 // 2:
                break
        return dict(kind="layer", mode=mode, M=M, K=K, N=Nn, bits=rng.choice((4, 6, 8)),
                    x=rng.choice(("relu", "outlier", "channels")),
                    g=rng.choice(("normal", "laplace")), sigma=rng.choice((1.5, 2.0, 2.5)))
    if kind == "quantize":
        C = _size(rng, 48, 11008)
        M = _size(rng, 256, min(200704, 16384 * 11008 // C))
        return dict(kind="quantize", M=M, C=C, bits=rng.choice((4, 6, 8)),
                    stochastic=rng.choice((True, False)), transposed=rng.choice((True, False)),
                    x=rng.choice(("relu", "outlier", "laplace")), sigma=2.0)
    if kind == "l1bn":
        C = _size(rng, 16, 2048)
        return dict(kind="l1bn", R=_size(rng, 3136, min(802816, 51380224 // C)), C=C,
                    bits=rng.choice((4, 8)))
    if kind == "pack":
        C = _size(rng, 64, 11008)
        return dict(kind="pack", M=_size(rng, 256, min(65536, 115605504 // C)), C=C,
                    bits=rng.choice((3, 4)))
    return dict(kind="chain", M=_size(rng, 64, 12608), K=_size(rng, 64, 1536),
                H=_size(rng, 64, 3072), N=_size(rng, 64, 1536), bits=rng.choice((4, 6)))


# ------------------------------------------------------------------------- inputs
def _tensor(recipe, rows, cols, gen, sigma=0.0):
    """fp32 [rows, cols]: post-ReLU activations, activations with a few outlier channels, or
    gradients whose channels differ widely in range (log-normal, a few far out)."""
    dev = gen.device
    if recipe == "relu":
        return torch.randn((rows, cols), generator=gen, device=dev).abs_()
    if recipe == "outlier":
        x = torch.randn((rows, cols), generator=gen, device=dev)
        n = max(1, round(0.02 * cols))
        x[:, torch.randperm(cols, generator=gen, device=dev)[:n]] *= 50.0
        return x
    if recipe == "weight":
        return torch.randn((rows, cols), generator=gen, device=dev).mul_(0.02)
    if recipe == "laplace":
        x = torch.empty((rows, cols), device=dev).exponential_(1.0, generator=gen)
        x -= torch.empty((rows, cols), device=dev).exponential_(1.0, generator=gen)
    else:  # "normal", "channels"
        x = torch.randn((rows, cols), generator=gen, device=dev)
    f = torch.randn(cols, generator=gen, device=dev).mul_(sigma or 1.5).exp_()
    n = max(1, round(0.005 * cols))
    f[torch.randperm(cols, generator=gen, device=dev)[:n]] *= 100.0
    return x.mul_(f)


def _inputs(case, seed):
    """The fp32 tensors the calls of a case take, from the seed alone."""
    gen = torch.Generator(device="cuda" if torch.cuda.is_available() else "cpu")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind == "layer":
        return {"x": _tensor(case["x"], case["M"], case["K"], gen, 1.5),
                "w": _tensor("weight", case["K"], case["N"], gen),
                "dy": _tensor(case["g"], case["M"], case["N"], gen, case["sigma"])}
    if kind == "quantize":
        return {"x": _tensor(case["x"], case["M"], case["C"], gen, case["sigma"])}
    if kind == "pack":
        return {"x": _tensor("relu", case["M"], case["C"], gen)}
    if kind == "l1bn":
        R, C = case["R"], case["C"]
        return {"x": _tensor("outlier", R, C, gen),
                "dy": _tensor("laplace", R, C, gen, 2.0),
                "gamma": torch.randn(C, generator=gen, device=gen.device).mul_(0.1).add_(1.0),
                "beta": torch.randn(C, generator=gen, device=gen.device).mul_(0.1)}
    return {"x": _tensor("outlier", case["M"], case["K"], gen),
            "w1": _tensor("weight", case["K"], case["H"], gen),
            "w2": _tensor("weight", case["H"], case["N"], gen),
            "dy": _tensor("laplace", case["M"], case["N"], gen, 2.0)}


def prepare(case, seed):
    t = _inputs(case, seed)
    kind, bits = case["kind"], case["bits"]
    dev = t["x"].device
    s = dict(t, case=case)
    if kind == "layer":
        mode = case["mode"]
        lay = L.QuantLinear(case["M"], case["K"], case["N"], bits, GROUPS, dev,
                            grouped=mode == "grouped", transposed=None)
        s["layer"] = lay
        if mode == "call":
            s["args"] = lay.step_args(t["x"], t["w"], t["dy"])
        elif mode == "graph":
            streams = [torch.cuda.Stream(device=dev) for _ in range(3)]
            s["graph"] = L.CapturedStep(
                lambda: lay.step_concurrent(t["x"], t["w"], t["dy"], SEED, streams))
    elif kind == "quantize":
        s["q"] = L.ShiftTensor.alloc(case["M"], case["C"], bits, GROUPS, dev, case["transposed"])
        s["status"] = torch.zeros(1, dtype=torch.int32, device=dev)
    elif kind == "l1bn":
        R, C = case["R"], case["C"]
        s["state"] = torch.zeros(N.shiftquant_l1bn_state_bytes(R, C), dtype=torch.uint8, device=dev)
        s["y"], s["dx"] = torch.zeros_like(t["x"]), torch.zeros_like(t["x"])
        s["dgamma"], s["dbeta"] = torch.zeros_like(t["gamma"]), torch.zeros_like(t["gamma"])
        s["status"] = torch.zeros(1, dtype=torch.int32, device=dev)
    elif kind == "pack":
        M, C = case["M"], case["C"]
        s["status"] = torch.zeros(1, dtype=torch.int32, device=dev)
        q = L.ShiftTensor.alloc(M, C, bits, GROUPS, dev, False)
        L.shift_quantize(s.pop("x"), q, bits, GROUPS, N.SQ_ROUND_NEAREST_EVEN, 0, s["status"])
        s["codes"], s["back"] = q.codes, L.empty_codes(M, C, bits, GROUPS, dev)
        s["packed"] = torch.zeros((M, (C + 1) // 2 + 15 & ~15), dtype=torch.uint8, device=dev)
    else:
        s["chain"] = ch = L.LinearChain(case["M"], (case["K"], case["H"], case["N"]), bits, GROUPS,
                                        dev)
        s["graph"] = L.CapturedStep(
            lambda: ch.step(t["x"], (t["w1"], t["w2"]), t["dy"], SEED))
    return s


def run(s):
    case = s["case"]
    kind, bits = case["kind"], case["bits"]
    if kind == "layer":
        lay = s["layer"]
        if case["mode"] == "call":
            N.shiftquant_layer_step(s["args"], SEED)
        elif case["mode"] == "graph":
            s["graph"].replay()
        else:
            lay.step(s["x"], s["w"], s["dy"], SEED)
        return {"y": lay.y, "dx": lay.dx, "dw": lay.dw, "x_exp": lay.x.exp, "g_exp": lay.g.exp}
    if kind == "quantize":
        q = s["q"]
        L.shift_quantize(s["x"], q, bits, GROUPS, int(case["stochastic"]), SEED, s["status"])
        out = {"codes": q.codes, "exp": q.exp, "range": q.range, "scale": q.scale}
        if q.codes_t is not None:
            out["codes_t"] = q.codes_t
        return out
    if kind == "l1bn":
        N.shiftquant_l1bn_forward(s["x"], s["gamma"], s["beta"], bits, GROUPS, s["y"], s["state"],
                                  s["status"])
        N.shiftquant_l1bn_backward(s["dy"], bits, GROUPS, SEED, s["state"], s["dx"], s["dgamma"],
                                   s["dbeta"], s["status"])
        return {"y": s["y"], "dx": s["dx"], "dgamma": s["dgamma"], "dbeta": s["dbeta"]}
    if kind == "pack":
        N.shiftquant_pack_codes(s["codes"], bits, GROUPS, s["packed"], s["status"])
        N.shiftquant_unpack_codes(s["packed"], case["C"], bits, GROUPS, s["back"])
        return {"packed": s["packed"], "back": s["back"]}
    ch = s["chain"]
    s["graph"].replay()
    return {"y": [lay.y for lay in ch.layers], "dx": [lay.dx for lay in ch.layers],
            "dw": [lay.dw for lay in ch.layers]}


def work(case):
    """Bytes (each input read once, each output written once) and operations of one pass."""
    kind = case["kind"]
    if kind == "layer":
        M, K, Nn = case["M"], case["K"], case["N"]
        return {"bytes": 2 * 4 * (M * K + K * Nn + M * Nn), "flops": 3 * 2 * M * K * Nn}
    code = 1 if case["bits"] <= 4 else 2
    if kind == "quantize":
        n = case["M"] * case["C"]
        return {"bytes": n * (4 + code * (2 if case["transposed"] else 1)), "flops": 0}
    if kind == "l1bn":
        return {"bytes": 4 * 4 * case["R"] * case["C"], "flops": 0}
    if kind == "pack":
        return {"bytes": 3 * case["M"] * case["C"], "flops": 0}
    M, K, H, Nn = case["M"], case["K"], case["H"], case["N"]
    # x, dy, both weights in; y, dx, dw of both layers out
    n = M * K + M * Nn + K * H + H * Nn + M * H + M * Nn + M * K + M * H + K * H + H * Nn
    return {"bytes": 4 * n, "flops": 3 * 2 * M * H * (K + Nn)}


# ------------------------------------------------------- the method's values in 64 bits
def _draws(rows, cols, seed, device):
    """The stochastic-rounding draws in [0, 1): the top 24 bits of SplitMix64's outputs."""
    def wrap(v):
        return v - (1 << 64) if v >= 1 << 63 else v

    def lsr(z, n):
        return (z >> n) & ((1 << (64 - n)) - 1)

    z = torch.arange(1, rows * cols + 1, dtype=torch.int64, device=device)
    z.mul_(wrap(0x9E3779B97F4A7C15)).add_(seed)
    z = (z ^ lsr(z, 30)) * wrap(0xBF58476D1CE4E5B9)
    z = (z ^ lsr(z, 27)) * wrap(0x94D049BB133111EB)
    return (lsr(z ^ lsr(z, 31), 40).double() * 2.0 ** -24).reshape(rows, cols)


def _shift(x, bits, seed=None):
    """codes, exponents, scale of a ShiftQuant tensor, in float64; rounded stochastically under
    `seed` where one is given."""
    Q = float(2 ** (bits - 1) - 1)
    x = x.double()
    r = x.abs().amax(0)
    tau = r.max()
    e = torch.zeros_like(r)
    for k in range(1, GROUPS):
        e = torch.where(r * 2.0 ** k <= tau, torch.full_like(e, k), e)
    v = x * 2.0 ** e * (Q / tau)
    if seed is not None:
        low = v.floor()
        q = low + (_draws(*x.shape, seed, x.device) < v - low)
    else:
        q = v.round()
    return q.clamp_(-Q, Q), e, tau / Q


def _channel(w, dim, bits):
    """codes and scales of a weight with one scale per column (dim 0) or per row (dim 1)."""
    Q = float(2 ** (bits - 1) - 1)
    w = w.double()
    r = w.abs().amax(dim, keepdim=True)
    return (w * (Q / r)).round(), r / Q


def _forward(qx, ex, sx, w, bits):
    q, s = _channel(w, 0, bits)
    return (qx * 2.0 ** -ex) @ q * (sx * s)


def _backward(qx, ex, sx, qg, eg, sg, w, bits):
    q, s = _channel(w, 1, bits)
    dx = (qg * 2.0 ** -eg) @ q.t() * (sg * s.t())
    dw = (qx * (sx * 2.0 ** -ex)).t() @ (qg * (sg * 2.0 ** -eg))
    return dx, dw


def _quant8(v):
    m = v.abs().max()
    return (v * (127.0 / m)).round().clamp_(-127, 127) * (m / 127.0)


def exact(case, seed):
    t = _inputs(case, seed)
    kind, bits = case["kind"], case["bits"]
    if kind == "pack":
        return None
    if kind == "layer":
        qx, ex, sx = _shift(t["x"], bits)
        y = _forward(qx, ex, sx, t["w"], bits)
        qg, eg, sg = _shift(t["dy"], bits, SEED)
        dx, dw = _backward(qx, ex, sx, qg, eg, sg, t["w"], bits)
        return {"y": y, "dx": dx, "dw": dw, "x_exp": None, "g_exp": None}
    if kind == "quantize":
        q, e, s = _shift(t["x"], bits, SEED if case["stochastic"] else None)
        codes = q if bits > 4 else None      # 4-bit codes are bytes, not numbers
        out = {"codes": codes, "exp": None, "range": t["x"].double().abs().amax(0),
               "scale": s.reshape(1)}
        if case["transposed"]:
            out["codes_t"] = None if codes is None else codes.t()
        return out
    if kind == "l1bn":
        q, e, s = _shift(t["x"], bits)
        step = s * 2.0 ** -e
        m = q.mean(0).round()
        d = q - m
        sigma = _quant8(d.abs().mean(0) * step)
        gamma, beta = _quant8(t["gamma"].double()), _quant8(t["beta"].double())
        on = sigma > 0
        inv = torch.where(on, 1.0 / sigma, torch.zeros_like(sigma))
        xhat = d * (step * inv)
        y = gamma * xhat + beta
        p, eg, sg = _shift(t["dy"], bits, SEED)
        g = p * (sg * 2.0 ** -eg)
        sign = d.sign()
        dgamma = (g * xhat).sum(0)
        dx = gamma * inv * (g - g.mean(0) - (g * xhat).mean(0) * (sign - sign.mean(0)))
        return {"y": y, "dx": dx, "dgamma": dgamma, "dbeta": g.sum(0)}
    # the chain: layer l draws its stochastic rounding under SEED + l
    q1, e1, s1 = _shift(t["x"], bits)
    y1 = _forward(q1, e1, s1, t["w1"], bits)
    q2, e2, s2 = _shift(y1, bits)
    y2 = _forward(q2, e2, s2, t["w2"], bits)
    g2, eg2, sg2 = _shift(t["dy"], bits, SEED + 1)
    dx2, dw2 = _backward(q2, e2, s2, g2, eg2, sg2, t["w2"], bits)
    g1, eg1, sg1 = _shift(dx2, bits, SEED)
    dx1, dw1 = _backward(q1, e1, s1, g1, eg1, sg1, t["w1"], bits)
    return {"y": [y1, y2], "dx": [dx1, dx2], "dw": [dw1, dw2]}

