"""Performance cases of the quantized linear and convolution path, through its public Python API.

Every case is one thing a program does with the library:

  linears     the quantized linears of transformer encoder blocks (QKV, proj, fc1, fc2): prologue + mixed GEMM per
              layer, at one low-bit ratio or over a sweep of them (run-time switch), launched call by call or
              replayed from one CUDA graph as a serving process keeps it
  linear      one linear layer of any shape, static or dynamic extraction positions
  conv        one convolution layer, NHWC
  bottleneck  1x1 -> ReLU -> 3x3 -> ReLU -> 1x1 with fused layer boundaries (no 8-bit tensor between the layers)
  calibrate   group order and extraction positions of a layer from calibration activations, on the device
  search      fitness of a few chromosomes of the group-selection search (layers laid out again for each)

Weights are a random-init 8-bit model; activations follow the distributions of `inputs.py` (Gaussian with 5 % of
channels x20 for linears, post-ReLU half-normal with per-channel ranges for convolutions), drawn on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_02822_b200 import binding as fx
from paper_2510_02822_b200 import calib, evolution

IN_TYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
OUT_MODES = {"i8": fx.OUT_REQUANT_I8, "f16": fx.OUT_DEQUANT_F16, "bf16": fx.OUT_DEQUANT_BF16, "f32": fx.OUT_DEQUANT_F32, "i32": fx.OUT_ACC_I32}
OUT_BYTES = {"i8": 1, "f16": 2, "bf16": 2, "f32": 4, "i32": 4}
IN_BYTES = {"f32": 4, "f16": 2, "bf16": 2}


def listed():
    return [
        # one small layer (DeiT-S proj, one image): the latency of a single call pair
        {"name": "linear_one_image", "kind": "linear", "rows": 197, "K": 384, "N": 384, "G": 16, "in": "f16", "out": "f16", "ratio": 0.5, "dynamic": False},
        # serving one request: the 48 linears of DeiT-S, one graph per (ratio, batch) as the serving experiment keeps it
        {"name": "serve_deits_b1", "kind": "linears", "rows": 197, "D": 384, "blocks": 12, "G": 16, "in": "f32", "out": "i8", "ratios": "0.5", "graph": True},
        # one encoder block's linears at a small batch, called one by one between 16-bit operators
        {"name": "block_deits_b8", "kind": "linears", "rows": 1576, "D": 384, "blocks": 1, "G": 16, "in": "f16", "out": "f16", "ratios": "0.25", "graph": False},
        # the benchmark's step: ViT-B linears, batch 64, every ratio in turn
        {"name": "sweep_vitb_b64", "kind": "linears", "rows": 12608, "D": 768, "blocks": 1, "G": 16, "in": "f32", "out": "i8", "ratios": "0,0.25,0.5,0.75,1", "graph": False},
        # the largest model's block: ViT-L, batch 128, 16-bit operators around the linears
        {"name": "block_vitl_b128", "kind": "linears", "rows": 25216, "D": 1024, "blocks": 1, "G": 16, "in": "f16", "out": "f16", "ratios": "0.75", "graph": False},
        # sizes that divide nothing: odd rows, K and N off the tile sizes, a ratio inside a K block
        {"name": "linear_ragged", "kind": "linear", "rows": 1001, "K": 720, "N": 1104, "G": 16, "in": "bf16", "out": "f32", "ratio": 0.3, "dynamic": False},
        # extraction positions found at run time on the widest ViT-B input
        {"name": "linear_dynamic", "kind": "linear", "rows": 12608, "K": 3072, "N": 768, "G": 16, "in": "f16", "out": "f16", "ratio": 0.5, "dynamic": True},
        # ResNet-50 convolutions at batch 32: the first stage, and a down-sampling one
        {"name": "conv3x3_56", "kind": "conv", "images": 32, "H": 56, "W": 56, "C": 64, "N": 64, "R": 3, "stride": 1, "G": 16, "in": "f32", "out": "i8", "ratio": 0.5},
        {"name": "conv3x3_28_s2", "kind": "conv", "images": 32, "H": 28, "W": 28, "C": 256, "N": 256, "R": 3, "stride": 2, "G": 16, "in": "f16", "out": "f16", "ratio": 0.5},
        # a ResNet-50 block with fused boundaries
        {"name": "bottleneck_14", "kind": "bottleneck", "images": 32, "H": 14, "W": 14, "C": 1024, "mid": 256, "G": 16, "in": "f16", "out": "i8", "ratio": 0.5},
        # calibration of a ViT-B linear on one batch
        {"name": "calibrate_vitb", "kind": "calibrate", "rows": 12608, "K": 768, "N": 3072, "G": 16, "in": "f32", "coverage": 0.0},
        # one step of the selection search: eight chromosomes on two ViT-B MLPs
        {"name": "search_vitb", "kind": "search", "rows": 1576, "D": 768, "blocks": 2, "G": 16, "ratio": 0.5, "chromosomes": 8},
    ]


def _log(rng, lo, hi, step=1):
    return max(lo, min(hi, step * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)))


def draw(rng):
    kind = rng.choice(["linear", "linear", "linears", "linears", "conv", "conv", "bottleneck", "calibrate", "search"])
    G = rng.choice([16, 16, 32])
    ratio = rng.choice([0.0, 0.25, 0.5, 0.75, 1.0, round(rng.uniform(0.05, 0.95), 2)])
    tin, tout = rng.choice(["f32", "f16", "bf16"]), rng.choice(["i8", "i8", "f16", "bf16", "f32"])
    if kind == "linear":
        c = {"kind": kind, "rows": _log(rng, 1, 25216), "K": _log(rng, 128, 4096, G), "N": _log(rng, 64, 4096, 16), "G": G, "in": tin, "out": tout,
             "ratio": ratio, "dynamic": rng.random() < 0.25}
    elif kind == "linears":
        graph = rng.random() < 0.5
        D = rng.choice([192, 384, 768, 1024])
        blocks = rng.choice([4, 12]) if graph else 1
        rows = _log(rng, 1, 8 if graph else 128) * 197
        c = {"kind": kind, "rows": rows, "D": D, "blocks": blocks, "G": G, "in": tin, "out": tout,
             "ratios": rng.choice(["0", "0.25", "0.5", "0.75", "1"]) if graph or rng.random() < 0.7 else "0,0.5,1", "graph": graph}
        while work(c)["flops"] > 6e11:
            c["rows"] = max(197, c["rows"] // 2)
    elif kind == "conv":
        side, C = rng.choice([(56, 64), (28, 128), (14, 256), (7, 512)])
        R = rng.choice([1, 3, 3])
        H, C = max(5, side + rng.randint(-2, 3)), C + rng.choice([0, 0, 16, -16]) * (G // 16)
        c = {"kind": kind, "images": _log(rng, 1, 64), "H": H, "W": H if rng.random() < 0.7 else max(5, H - rng.randint(1, 4)), "C": C,
             "N": C * (4 if R == 1 and rng.random() < 0.6 else 1), "R": R, "stride": rng.choice([1, 1, 2]) if R == 3 else 1, "G": G, "in": tin, "out": tout, "ratio": ratio}
    elif kind == "bottleneck":
        H, mid = rng.choice([(56, 64), (28, 128), (14, 256), (7, 512)])
        c = {"kind": kind, "images": _log(rng, 1, 64), "H": H, "W": H, "C": 4 * mid, "mid": mid, "G": G, "in": tin, "out": tout, "ratio": ratio}
    elif kind == "calibrate":
        c = {"kind": kind, "rows": _log(rng, 256, 25216), "K": _log(rng, 128, 4096, G), "N": _log(rng, 128, 4096, 16), "G": G, "in": tin,
             "coverage": rng.choice([0.0, 0.99])}
    else:
        c = {"kind": kind, "rows": 197 * _log(rng, 1, 16), "D": rng.choice([384, 768]), "blocks": rng.choice([1, 2]), "G": G,
             "ratio": rng.choice([0.25, 0.5, 0.75]), "chromosomes": rng.randint(4, 12)}
    return c


# ---------------------------------------------------------------------------------------------- inputs
class _Draw:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device="cuda")

    def uniform(self, *shape):
        return torch.rand(shape, generator=self.g, device="cuda")

    def ranges(self, n):                                   # log-uniform over [0.05, 8]
        return torch.exp(math.log(0.05) + self.uniform(n) * math.log(160.0))

    def activations(self, rows, K, half=False):
        """[rows, K] activations and a scale from a separate 256-row draw (also returned)."""
        ch = self.ranges(K) if half else torch.where(self.uniform(K) < 0.05, 20.0, 1.0)
        x, cal = self.normal(rows, K) * ch, self.normal(256, K) * ch
        if half:
            x, cal = x.abs_(), cal.abs_()
        return x, cal, float(np.float32(float(cal.abs().max()) / 127.0))

    def weights(self, w, out_axis):
        """Random-init 8-bit model: per-output-channel scale = absmax / 127."""
        red = [i for i in range(w.dim()) if i != out_axis]
        s = w.abs().amax(dim=red, keepdim=True) / 127.0
        return torch.clamp(torch.round(w / s), -127, 127).to(torch.int8).contiguous(), s.reshape(-1).contiguous()


def _linear_inputs(d, rows, K, N):
    x, cal, xs = d.activations(rows, K)
    Wq, ws = d.weights(d.normal(K, N) * 0.02, 1)
    bias = d.normal(N) * 0.02
    y = torch.clamp(torch.round(cal / xs), -128, 127) @ Wq.float() * (xs * ws) + bias
    return x, cal, xs, Wq, ws, bias, float(np.float32(float(y.abs().max()) / 127.0))


def _linear(d, rows, K, N, G, in_type):
    x, cal, xs, Wq, ws, bias, ys = _linear_inputs(d, rows, K, N)
    perm, shift, _ = calib.static_preparation_device(cal, xs, Wq, G)
    return {"layer": fx.Layer(Wq, ws, bias, perm, shift, G), "X": x.to(in_type), "xs": xs, "ys": ys, "rows": rows}


def _conv_weights(d, C, N, R):
    w = d.normal(N, R, R, C) * math.sqrt(2.0 / (R * R * C))
    Wq, ws = d.weights(w, 0)
    return Wq, ws, d.normal(N) * 0.1


def prepare(case, seed):
    d = _Draw(seed)
    G, kind = case["G"], case["kind"]
    if kind == "linear":
        s = _linear(d, case["rows"], case["K"], case["N"], G, IN_TYPES[case["in"]])
        s["layer"].set_lowbit_ratio(case["ratio"])
        return {"case": case, **s}
    if kind == "linears":
        D = case["D"]
        layers = [_linear(d, case["rows"], K, N, G, IN_TYPES[case["in"]])
                  for _ in range(case["blocks"]) for K, N in ((D, 3 * D), (D, D), (D, 4 * D), (4 * D, D))]
        s = {"case": case, "layers": layers, "ratios": [float(r) for r in case["ratios"].split(",")]}
        if case["graph"]:
            for l in layers:
                l["layer"].set_lowbit_ratio(s["ratios"][0])
                l["Y"] = torch.empty((l["rows"], l["layer"].N), dtype={1: torch.int8, 2: torch.float16, 4: torch.float32}[OUT_BYTES[case["out"]]]
                                     if case["out"] != "bf16" else torch.bfloat16, device="cuda")
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.stream(side):
                for l in layers:
                    _forward(l, OUT_MODES[case["out"]], l["Y"])
                side.synchronize()
                with torch.cuda.graph(s["graph"], stream=side):
                    for l in layers:
                        _forward(l, OUT_MODES[case["out"]], l["Y"])
            torch.cuda.current_stream().wait_stream(side)
        return s
    if kind == "conv":
        x, cal, xs = d.activations(case["images"] * case["H"] * case["W"], case["C"], half=True)
        Wq, ws, bias = _conv_weights(d, case["C"], case["N"], case["R"])
        perm, shift, _ = calib.static_preparation_device(cal, xs, Wq, G, conv=True)
        L = fx.Layer(Wq, ws, bias, perm, shift, G, conv=(case["stride"], case["R"] // 2))
        L.set_lowbit_ratio(case["ratio"])
        return {"case": case, "layer": L, "X": x.to(IN_TYPES[case["in"]]), "xs": xs, "ys": _conv_scale(cal, xs, Wq, ws, bias)}
    if kind == "bottleneck":
        rows = case["images"] * case["H"] * case["W"]
        x, cal, xs = d.activations(rows, case["C"], half=True)
        shapes = [(case["C"], case["mid"], 1), (case["mid"], case["mid"], 3), (case["mid"], case["C"], 1)]
        layers, scales, h = [], [xs], cal
        for C, N, R in shapes:
            Wq, ws, bias = _conv_weights(d, C, N, R)
            perm, shift, _ = calib.static_preparation_device(h, scales[-1], Wq, G, conv=True)
            layers.append((Wq, ws, bias, perm, shift, R))
            scales.append(_conv_scale(h, scales[-1], Wq, ws, bias))
            h = torch.relu(d.normal(256, N)) * (scales[-1] * 30.0)      # stands for the layer's post-ReLU outputs
        made = []
        for i, (Wq, ws, bias, perm, shift, R) in enumerate(layers):
            if i + 1 < len(layers):  # the next layer's channel order is moved into this layer's outputs, as a deployment does offline
                Wq, ws, bias = calib.permute_outputs_for_next(Wq, ws, bias, layers[i + 1][3], G, conv=True)
            made.append(fx.Layer(Wq, ws, bias, perm, shift, G, conv=(1, R // 2)))
            made[-1].set_lowbit_ratio(case["ratio"])
        return {"case": case, "layers": made, "X": x.to(IN_TYPES[case["in"]]), "scales": scales}
    if kind == "calibrate":
        x, _, xs = d.activations(case["rows"], case["K"])
        Wq, _ = d.weights(d.normal(case["K"], case["N"]) * 0.02, 1)
        return {"case": case, "X": x.to(IN_TYPES[case["in"]]), "xs": xs, "Wq": Wq}
    # search: fc1 -> fc2 pairs chained, int8 between the layers
    D, dims = case["D"], [case["D"]]
    for _ in range(case["blocks"]):
        dims += [4 * D, D]
    h, cal, xs = d.activations(case["rows"], D)
    X, layers, scores = h.cpu().numpy(), [], []
    for K, N in zip(dims[:-1], dims[1:]):
        Wq, ws = d.weights(d.normal(K, N) * 0.02, 1)
        bias = d.normal(N) * 0.02
        _, shift, info = calib.static_preparation_device(cal, xs, Wq, G)
        scores += info["score"].cpu().tolist()
        cal = torch.clamp(torch.round(cal / xs), -128, 127) @ Wq.float() * (xs * ws) + bias
        ys = float(np.float32(float(cal.abs().max()) / 127.0))
        layers.append(dict(Wq=Wq.cpu().numpy(), w_scale=ws.cpu().numpy(), bias=bias.cpu().numpy(), x_scale=xs, y_scale=ys, G=G, sx_group=shift))
        xs = ys
    fit = evolution.ChainFitness(layers, X, torch.device("cuda", torch.cuda.current_device()))
    target = [math.ceil(case["ratio"] * g - 1e-4) for g in fit.groups]
    pop, _ = fx.flexiq_evo_init(fit.groups, np.asarray(scores), target, case["chromosomes"], seed)
    return {"case": case, "fit": fit, "pop": pop}


def _conv_scale(cal, xs, Wq, ws, bias):
    """Output scale of a convolution from its centre tap, widened by the filter size."""
    R = Wq.shape[1]
    q = torch.clamp(torch.round(cal / xs), -128, 127)
    y = q @ Wq[:, R // 2, R // 2, :].T.float() * (xs * ws) + bias
    return float(np.float32(float(y.abs().max()) * R / 127.0))


# ---------------------------------------------------------------------------------------------- one pass
def _forward(l, mode, Y=None):
    x4, x8, _ = l["layer"].quantize_lower(l["X"], l["xs"])
    return l["layer"].mixed_gemm(x4, x8, l["rows"], l["xs"], l["ys"], mode, Y)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "linears":
        if case["graph"]:
            state["graph"].replay()
            return [l["Y"] for l in state["layers"]]
        out = []
        for ratio in state["ratios"]:
            for l in state["layers"]:
                l["layer"].set_lowbit_ratio(ratio)
                out.append(_forward(l, OUT_MODES[case["out"]]))
        return out
    if kind == "linear":
        if not case["dynamic"]:
            return _forward(state, OUT_MODES[case["out"]])
        x4, x8, pos = state["layer"].quantize_lower(state["X"], state["xs"], dynamic=True)
        return state["layer"].mixed_gemm(x4, x8, case["rows"], state["xs"], state["ys"], OUT_MODES[case["out"]], x_shift=pos), pos
    if kind == "conv":
        x4, x8, _ = state["layer"].quantize_lower(state["X"], state["xs"])
        return state["layer"].mixed_conv(x4, x8, case["images"], case["H"], case["W"], state["xs"], state["ys"], OUT_MODES[case["out"]])
    if kind == "bottleneck":
        a, b, c = state["layers"]
        shape, (s0, s1, s2, s3) = (case["images"], case["H"], case["W"]), state["scales"]
        x4, x8, _ = a.quantize_lower(state["X"], s0)
        h1 = a.mixed_conv_to_slab(x4, x8, *shape, s0, b, s1, relu=True, out_order=fx.ORDER_NEXT_SLAB)
        h2 = b.mixed_conv_to_slab(h1, None, *shape, s1, c, s2, relu=True, out_order=fx.ORDER_NEXT_SLAB)
        return c.mixed_conv(h2, None, *shape, s2, s3, OUT_MODES[case["out"]])
    if kind == "calibrate":
        perm, shift, info = calib.static_preparation_device(state["X"], state["xs"], state["Wq"], case["G"], coverage=case["coverage"] or None)
        return perm, shift, info
    dist = state["fit"].distances(state["pop"])
    return dist, state["fit"].Y[-1]


# ---------------------------------------------------------------------------------------------- the same in 64 bits
def _bits(lo, hi):
    """Lowest bit position that keeps four bits of every integer in [lo, hi] (lo <= 0 <= hi)."""
    m = torch.maximum(hi, -lo - 1)
    return sum((m >= 8 << b).long() for b in range(4))


def _quantized(x, xs):
    scale = torch.full((), xs, dtype=torch.float32, device=x.device)      # a tensor: a scalar divisor becomes a multiplication
    return torch.clamp(torch.round(x.float() / scale), -128, 127).double()


def _positions(q, Wmax, G):
    """Order of the channel groups (ascending activation range x weight range) and their positions, from quantized rows."""
    lo, hi = q.amin(0).clamp(max=0), q.amax(0).clamp(min=0)
    score = (torch.maximum(hi, -lo) * Wmax).reshape(-1, G).amax(1)
    return torch.sort(score, stable=True).indices, _bits(lo, hi).reshape(-1, G).amax(1)


def _lowered(v, s):
    """Integers v clipped to what four bits hold at position s, with the bits below it cleared."""
    return torch.floor(torch.minimum(torch.maximum(v, -(8 << s).double()), ((8 << s) - 1).double()) / (1 << s).double()) * (1 << s).double()


def _operands(x, cal, xs, W, G, ratio, dynamic=False):
    """8-bit activations [rows, K] and weights [taps, K, N] with the selected groups at 4 bits; the positions in slab order."""
    q = _quantized(x, xs)
    n_g = W.shape[1] // G
    order, pos = _positions(_quantized(cal, xs), W.abs().amax((0, 2)), G)
    if dynamic:
        pos = _bits(q.amin(0).clamp(max=0), q.amax(0).clamp(min=0)).reshape(-1, G).amax(1)
    low = torch.zeros(n_g, dtype=torch.bool, device=q.device)
    low[order[:math.ceil(ratio * n_g - 1e-4)]] = True
    ch = low.repeat_interleave(G)
    Wg = W.reshape(W.shape[0], n_g, G, -1)
    sw = _bits(Wg.amin((0, 2)).clamp(max=0), Wg.amax((0, 2)).clamp(min=0))
    q = torch.where(ch, _lowered(q, pos.repeat_interleave(G)), q)
    return q, torch.where(ch[None, :, None], _lowered(W, sw.repeat_interleave(G, 0)[None]), W), pos[order].to(torch.uint8)


def _finished(acc, case, xs, ws, bias, ys):
    if case["out"] == "i32":
        return acc
    y = acc.mul_(xs * ws.double()).add_(bias.double())
    return torch.clamp(torch.round(y / ys), -128, 127) if case["out"] == "i8" else y


def exact(case, seed):
    """Sums and scaling in 64 bits (Eq. 1's division is fp32 by definition); the other kinds return integers throughout."""
    d = _Draw(seed)
    G, kind = case["G"], case["kind"]
    if kind in ("linear", "linears"):
        D, out = case.get("D"), []
        shapes = [(case["K"], case["N"])] if kind == "linear" else [(D, 3 * D), (D, D), (D, 4 * D), (4 * D, D)] * case["blocks"]
        inputs = [_linear_inputs(d, case["rows"], K, N) for K, N in shapes]
        for ratio in ([case["ratio"]] if kind == "linear" else [float(r) for r in case["ratios"].split(",")]):
            for x, cal, xs, Wq, ws, bias, ys in inputs:
                q, W, pos = _operands(x.to(IN_TYPES[case["in"]]), cal, xs, Wq.double()[None], G, ratio, case.get("dynamic", False))
                out.append(_finished(q @ W[0], case, xs, ws, bias, ys))
        if kind == "linears":
            return out if sum(y.numel() for y in out) < 2.5e9 else None
        return (out[0], pos) if case["dynamic"] else out[0]
    if kind == "conv":
        R, stride, H, W_ = case["R"], case["stride"], case["H"], case["W"]
        x, cal, xs = d.activations(case["images"] * H * W_, case["C"], half=True)
        Wq, ws, bias = _conv_weights(d, case["C"], case["N"], R)
        taps = Wq.double().permute(1, 2, 3, 0).reshape(R * R, case["C"], case["N"])
        q, W, _ = _operands(x.to(IN_TYPES[case["in"]]), cal, xs, taps, G, case["ratio"])
        p = R // 2
        q = torch.nn.functional.pad(q.reshape(case["images"], H, W_, case["C"]), (0, 0, p, p, p, p))
        P, Q = (H + 2 * p - R) // stride + 1, (W_ + 2 * p - R) // stride + 1
        acc = sum(q[:, t // R:t // R + (P - 1) * stride + 1:stride, t % R:t % R + (Q - 1) * stride + 1:stride] @ W[t] for t in range(R * R))
        return _finished(acc, case, xs, ws, bias, _conv_scale(cal, xs, Wq, ws, bias))
    return None


# ---------------------------------------------------------------------------------------------- work and tolerance
def _gemm_work(M, K, N, ratio, in_bytes, out_bytes, taps=1):
    """X read once, W once (the low-bit part at 4 bits), Y written once."""
    return M * K * in_bytes + taps * K * N * (1 - ratio / 2) + 8 * N + M * N * out_bytes, 2.0 * M * K * N * taps


def work(case):
    kind = case["kind"]
    b = f = 0.0
    if kind == "linear":
        b, f = _gemm_work(case["rows"], case["K"], case["N"], case["ratio"], IN_BYTES[case["in"]], OUT_BYTES[case["out"]])
    elif kind == "linears":
        D = case["D"]
        for r in case["ratios"].split(","):
            for K, N in ((D, 3 * D), (D, D), (D, 4 * D), (4 * D, D)):
                x, y = _gemm_work(case["rows"], K, N, float(r), IN_BYTES[case["in"]], OUT_BYTES[case["out"]])
                b, f = b + case["blocks"] * x, f + case["blocks"] * y
    elif kind == "conv":
        P, Q = ((v + 2 * (case["R"] // 2) - case["R"]) // case["stride"] + 1 for v in (case["H"], case["W"]))
        M, pixels = case["images"] * P * Q, case["images"] * case["H"] * case["W"]
        b, f = _gemm_work(M, case["C"], case["N"], case["ratio"], 0, OUT_BYTES[case["out"]], case["R"] ** 2)
        b += pixels * case["C"] * IN_BYTES[case["in"]]
    elif kind == "bottleneck":
        M, C, mid, r = case["images"] * case["H"] * case["W"], case["C"], case["mid"], case["ratio"]
        for K, N, taps, i, o in ((C, mid, 1, IN_BYTES[case["in"]], 0), (mid, mid, 9, 0, 0), (mid, C, 1, 0, OUT_BYTES[case["out"]])):
            x, y = _gemm_work(M, K, N, r, i, o, taps)
            b, f = b + x, f + y
    elif kind == "calibrate":
        b = case["rows"] * case["K"] * IN_BYTES[case["in"]] + case["K"] * case["N"]
    else:  # per chromosome and layer: the weights laid out again (read once, written once) and one pass of the chain
        D, M, layers = case["D"], case["rows"], 2 * case["blocks"]
        b = case["chromosomes"] * (layers * 4 * D * D * (2 - case["ratio"] / 2) + M * D * (4 + 1))
        f = case["chromosomes"] * layers * 2.0 * M * 4 * D * D
    return {"bytes": b, "flops": f}


def tolerance(case):
    """Integers are exact.  Floating outputs are the exact int32 sum scaled in fp32 and rounded once to the output type:
    measured against float64, relative 2-norm errors of 5e-8 (fp32), 2e-4 (fp16) and 1.7e-3 (bf16)."""
    return {"f32": {"rel": 2e-7, "max": 1e-6}, "f16": {"rel": 8e-4, "max": 2e-3}, "bf16": {"rel": 6.5e-3, "max": 1.6e-2}}.get(case.get("out"), "exact")
