"""The measured workloads of this framework: the calls its users make, through the public entry
points (paper_1607_04683_gb300.qnn and .qat), over the sizes they make them at.

Kinds:
  quantize  qnn.qnn_quantize on fp32 rows in device memory: activations on the fly, one unit per
            row (layer inputs, frames of many sequences), or a whole matrix as one unit (weights
            offline, and again at every step of quantization-aware training).
  qmatmul   qnn.qnn_qmatmul on codes in device memory: one fully connected 8-bit layer, from one
            frame of one sequence to a large batch of frames.
  lstm      qnn.LstmModel.forward: a whole quantized LSTM / LSTMP acoustic model over a batch of
            sequences; device frames in, posteriors (or top-layer outputs) and final states out.
  linear    qat.QuantLinear: one training step of a fully connected layer, forward (quantized) and
            backward (full precision), gradients out.

The model shapes are the package's own synthetic workloads (inputs.py: 5 x 500 cells with 2000
classes, 5 x 2048 cells with a 512-unit projection and 8192 classes) and the Sec. 4 frontend (8
stacked frames of 40 features, every third kept), the products those of its matrix-product sweep.
"""
from __future__ import annotations

import math

import torch

from paper_1607_04683_gb300 import qat, qnn

DEV = "cuda"


# ------------------------------------------------------------------------------------------------
# The cases
# ------------------------------------------------------------------------------------------------

def _lstm(name=None, layers=5, dim=40, hidden=500, proj=0, classes=2000, mode="quant", stack=1, stride=1, batch=1,
          frames=100, wrange=0.08, states=False, blocks=1):
    c = {"kind": "lstm", "layers": layers, "dim": dim, "hidden": hidden, "proj": proj, "classes": classes,
         "mode": mode, "stack": stack, "stride": stride, "batch": batch, "frames": frames, "wrange": wrange,
         "states": states, "blocks": blocks}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the layer input of a batch of utterances, quantized on the fly, one unit per frame
        {"name": "quantize_rows_128000x500", "kind": "quantize", "rows": 128000, "cols": 500, "pad": 0,
         "per_row": True},
        # a large weight matrix as one unit
        {"name": "quantize_matrix_8192x8192", "kind": "quantize", "rows": 8192, "cols": 8192, "pad": 0,
         "per_row": False},
        # one frame through one layer: the smallest product, bound by latency
        {"name": "qmatmul_m1_2048", "kind": "qmatmul", "m": 1, "n": 2048, "k": 2048, "per_row": False, "blocks": 1,
         "bias": True, "acc": False},
        # a second of frames through the output layer of the 500-cell model (odd sizes)
        {"name": "qmatmul_m100_2000x500", "kind": "qmatmul", "m": 100, "n": 2000, "k": 500, "per_row": True,
         "blocks": 1, "bias": True, "acc": False},
        # a batch of frames through a large layer, raw accumulators returned too
        {"name": "qmatmul_m256_8192", "kind": "qmatmul", "m": 256, "n": 8192, "k": 8192, "per_row": True,
         "blocks": 4, "bias": True, "acc": True},
        # the largest product of the sweep
        {"name": "qmatmul_m16384_8192", "kind": "qmatmul", "m": 16384, "n": 8192, "k": 8192, "per_row": False,
         "blocks": 1, "bias": False, "acc": False},
        # one utterance, the embedded setting
        _lstm("lstm_5x500_b1", batch=1, frames=300),
        # a server's batch of streams, a chunk of frames at a time, with carried states
        _lstm("lstm_5x500_b16_chunk", batch=16, frames=100, states=True),
        # stacked frames and the float output layer ("quant")
        _lstm("lstm_5x500_b64_stack_float", batch=64, frames=300, stack=8, stride=3, mode="float"),
        # offline transcription, a batch of utterances
        _lstm("lstm_5x500_b256", batch=256, frames=500),
        # the large projected model at its full batch
        _lstm("lstmp_5x2048p512_b1024", dim=80, hidden=2048, proj=512, classes=8192, batch=1024, frames=100,
              wrange=0.05),
        # one training step of a fully connected layer
        {"name": "linear_4096x512x2048", "kind": "linear", "m": 4096, "k": 512, "n": 2048, "bias": True},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["quantize", "quantize", "qmatmul", "qmatmul", "qmatmul", "lstm", "lstm", "lstm", "linear"])
    if kind == "quantize":
        per_row = rng.random() < 0.6
        cols = _log(rng, 17, 8192)
        rows = _log(rng, 1, min(200000, (1 << 26) // cols))
        return {"kind": kind, "rows": rows, "cols": cols, "pad": rng.choice([0, 0, 0, 4, 7]), "per_row": per_row}
    if kind == "qmatmul":
        blocks = rng.choice([1, 1, 1, 4])
        n = max(blocks, _log(rng, 64, 8192) // blocks * blocks)
        return {"kind": kind, "m": _log(rng, 1, 16384), "n": n, "k": _log(rng, 40, 8192),
                "per_row": rng.random() < 0.5, "blocks": blocks, "bias": rng.random() < 0.5,
                "acc": rng.random() < 0.2}
    if kind == "linear":
        return {"kind": kind, "m": _log(rng, 16, 8192), "k": _log(rng, 40, 1024), "n": _log(rng, 64, 2048),
                "bias": rng.random() < 0.8}
    if rng.random() < 0.3:  # projected models
        hidden = rng.choice([512, 800, 1024, 2048])
        return _lstm(layers=rng.randint(1, 5), dim=rng.choice([40, 80]), hidden=hidden,
                     proj=rng.choice([100, 128, 200, 256, 512]), classes=rng.choice([0, 2000, 8192]),
                     batch=_log(rng, 64, 1024), frames=rng.randint(8, 60), wrange=0.05, states=rng.random() < 0.3)
    hidden = rng.choice([128, 300, 301, 400, 450, 500, 512])
    stack = rng.choice([1, 1, 8])
    blocks = rng.choice([1, 1, 1, 4]) if hidden % 16 == 0 else 1
    mode = "float" if rng.random() < 0.25 else "quant"
    classes = rng.choice([0, 999, 2000, 4000])
    if blocks > 1 and classes == 999:
        classes = 1000
    return _lstm(layers=rng.randint(1, 5), hidden=hidden, classes=classes, mode=mode, stack=stack,
                 stride=3 if stack > 1 else 1, batch=_log(rng, 1, 256), frames=_log(rng, 10, 150),
                 states=rng.random() < 0.3, blocks=blocks)


# ------------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _normal(g, *shape, std=1.0):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32) * std


def _uniform(g, *shape, a=1.0):
    return (torch.rand(shape, generator=g, device=DEV, dtype=torch.float32) * 2 - 1) * a


def _quantize_input(case, seed):
    g = _gen(seed)
    x = _normal(g, case["rows"], case["cols"] + case["pad"])
    if case["per_row"]:  # layer outputs and frames: each row with its own mean and spread
        x = x * (0.2 + torch.rand((case["rows"], 1), generator=g, device=DEV)) + _uniform(g, case["rows"], 1, a=0.5)
    else:
        x = x * 0.05
    return x[:, :case["cols"]]


def _qmatmul_input(case, seed):
    """Weights ~ N(0, 0.05), activations sigmoid(N(0, 2)) (gate outputs), bias ~ U(-0.1, 0.1)."""
    g = _gen(seed)
    w = _normal(g, case["n"], case["k"], std=0.05)
    a = torch.sigmoid(_normal(g, case["m"], case["k"], std=2.0))
    b = _uniform(g, case["n"], a=0.1) if case["bias"] else None
    return w, a, b


def _lstm_sizes(case):
    R = case["proj"] if case["proj"] > 0 else case["hidden"]
    return case["layers"], case["dim"] * case["stack"], case["hidden"], case["proj"], case["classes"], R


def _lstm_input(case, seed):
    """The packed parameters as a list of tensors (per layer Wx[4], Wh[4], b, Wp; then Wo, bo), the
    frames [B, T, dim] with a mean offset per sequence, and initial states where the case has them."""
    L, I, H, P, C, R = _lstm_sizes(case)
    g = _gen(seed)
    a = case["wrange"]
    parts = []
    for l in range(L):
        parts.append(_uniform(g, 4, H, I if l == 0 else R, a=a))
        parts.append(_uniform(g, 4, H, R, a=a))
        b = torch.zeros((4, H), device=DEV)
        b[1] = 1.0
        parts.append(b)
        if P > 0:
            parts.append(_uniform(g, P, H, a=a))
    if C > 0:
        parts.append(_uniform(g, C, R, a=0.5))  # spread logits
        parts.append(torch.zeros(C, device=DEV))
    B, T = case["batch"], case["frames"]
    x = _normal(g, B, T, case["dim"]) + _uniform(g, B, 1, 1, a=0.5)
    h = c = None
    if case["states"]:
        h, c = _uniform(g, L, B, R, a=0.5), _normal(g, L, B, H, std=0.5)
    return parts, x, h, c


def prepare(case, seed):
    kind = case["kind"]
    if kind == "quantize":
        return {"case": case, "x": _quantize_input(case, seed)}
    if kind == "qmatmul":
        w, a, b = _qmatmul_input(case, seed)
        per = case["n"] // case["blocks"]
        q = [qnn.qnn_quantize(w[i * per:(i + 1) * per], qnn.PER_MATRIX) for i in range(case["blocks"])]
        cw, pw, sw = (torch.cat([p[j] for p in q]) for j in range(3))
        ga = qnn.PER_ROW if case["per_row"] else qnn.PER_MATRIX
        ca, pa, sa = qnn.qnn_quantize(a, ga)
        return {"case": case, "A": ca, "pa": pa, "ga": ga, "rsA": sa, "W": cw, "pw": pw, "csW": sw, "bias": b}
    if kind == "lstm":
        parts, x, h, c = _lstm_input(case, seed)
        mode = {"quant": qnn.OUT_QUANT, "float": qnn.OUT_FLOAT}[case["mode"]] if case["classes"] > 0 else qnn.OUT_NONE
        d = qnn.lstm_desc(case["layers"], case["dim"], case["hidden"], case["proj"], case["classes"], mode,
                          stack=case["stack"], stack_stride=case["stride"], weight_blocks=case["blocks"])
        model = qnn.LstmModel(d, torch.cat([p.reshape(-1) for p in parts]))
        return {"case": case, "model": model, "x": x, "h": h, "c": c}
    g = _gen(seed)
    layer = qat.QuantLinear(case["k"], case["n"], bias=case["bias"], device=DEV)
    with torch.no_grad():
        layer.weight.copy_(_uniform(g, case["n"], case["k"], a=case["k"] ** -0.5))
        if case["bias"]:
            layer.bias.copy_(_uniform(g, case["n"], a=0.1))
    x = torch.sigmoid(_normal(g, case["m"], case["k"], std=2.0)).requires_grad_()
    return {"case": case, "layer": layer, "x": x, "g": _normal(g, case["m"], case["n"], std=1e-3)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "quantize":
        return qnn.qnn_quantize(state["x"], qnn.PER_ROW if case["per_row"] else qnn.PER_MATRIX)
    if kind == "qmatmul":
        return qnn.qnn_qmatmul(state["A"], state["pa"], state["ga"], state["rsA"], state["W"], state["pw"],
                               state["csW"], n_blocks=case["blocks"], bias=state["bias"], want_acc=case["acc"])
    if kind == "lstm":
        y = state["model"].forward(state["x"], h_state=state["h"], c_state=state["c"])
        return {"y": y, "h": state["h"], "c": state["c"]}
    layer, x = state["layer"], state["x"]
    x.grad = layer.weight.grad = None
    if case["bias"]:
        layer.bias.grad = None
    y = layer(x)
    y.backward(state["g"])
    return {"y": y.detach(), "gx": x.grad, "gw": layer.weight.grad, "gb": layer.bias.grad if case["bias"] else None}


# ------------------------------------------------------------------------------------------------
# What a pass cannot do without
# ------------------------------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "quantize":
        n = case["rows"] * case["cols"]
        return {"bytes": 5 * n + 4 * case["rows"] + 16 * (case["rows"] if case["per_row"] else 1), "flops": 0}
    if kind == "qmatmul":
        m, n, k = case["m"], case["n"], case["k"]
        out = 4 * m * n * (2 if case["acc"] else 1)
        return {"bytes": m * k + n * k + out + 20 * m + 8 * n, "flops": 2 * m * n * k}
    if kind == "lstm":
        L, I, H, P, C, R = _lstm_sizes(case)
        B, T = case["batch"], case["frames"]
        Tn = (T + case["stride"] - 1) // case["stride"]
        wb = sum(4 * H * ((I if l == 0 else R) + R) + 16 * H + P * H for l in range(L))
        fl = B * Tn * sum(2 * (4 * H * ((I if l == 0 else R) + R) + P * H) for l in range(L))
        if C > 0:
            wb += C * R * (4 if case["mode"] == "float" else 1) + 4 * C
            fl += 2 * B * Tn * C * R
        st = 4 * 2 * L * B * (R + H) if case["states"] else 0
        return {"bytes": wb + 4 * B * T * case["dim"] + 4 * B * Tn * (C if C > 0 else R) + st, "flops": fl}
    m, n, k = case["m"], case["n"], case["k"]
    return {"bytes": 4 * (2 * m * k + 2 * n * k + 2 * m * n), "flops": 6 * m * n * k}


def tolerance(case):
    """Codes, unit parameters and code sums are whole numbers and exact. The products are exact
    integers recovered by a few 32-bit operations, measured 4e-8 to 6e-8 from 64 bits; a softmax
    adds a 32-bit sum of its terms in any order and the float output layer a 32-bit dot product.
    The training step's gradients are 32-bit products of any order."""
    kind = case["kind"]
    if kind == "quantize":
        return "exact"
    if kind == "qmatmul":
        return {"rel": 5e-7, "max": 5e-6}
    if kind == "lstm":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 5e-6, "max": 1e-4}


# ------------------------------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ------------------------------------------------------------------------------------------------

def _units(v, dim):
    """Q and z of the quantizer's definition (its fp32 steps) for the ranges of v over `dim`."""
    v = v.float()
    mn, mx = (v.amin(dim, keepdim=True), v.amax(dim, keepdim=True))
    big, s = 4194304.0, torch.full_like(mn, 255.0)
    R = mx - mn
    Q = s / R
    deg = ~(R > 0) | ~torch.isfinite(Q) | ~((Q * mn).abs() < big) | ~((Q * mx).abs() < big)
    amax = torch.maximum(mn.abs(), mx.abs())
    Qd = torch.where(amax > 0, s / amax, torch.ones_like(s))
    Q = torch.where(deg, Qd, Q)
    up = torch.full_like(Q, math.inf)
    for _ in range(64):
        short = ~deg & (torch.round(Q * mx) - torch.round(Q * mn) < 255)
        if not bool(short.any()):
            break
        Q = torch.where(short, torch.nextafter(Q, up), Q)
    return Q, torch.round(Q * mn)


def _offset_codes(v, dim):
    """(codes + z) of eq. (1) in 64 bits, and Q."""
    v = v.float()
    Q, z = _units(v, dim)
    c = (torch.round(Q * v) - z).clamp(0, 255)
    return (c + z).double(), Q.double()


def _weights(w, blocks):
    """[rows, cols] -> (codes + z) [rows, cols] and Q [rows], one unit per block of rows."""
    n, k = w.shape
    a, Q = _offset_codes(w.reshape(blocks, -1), 1)
    return a.reshape(n, k), Q.expand(blocks, n // blocks).reshape(-1)


def _layer(x, w, Qw):
    a, Qa = _offset_codes(x, -1)
    return (a @ w.t()) / (Qa * Qw)


def _lstm_exact(case, seed):
    parts, x, h0, c0 = _lstm_input(case, seed)
    L, I, H, P, C, R = _lstm_sizes(case)
    B, T, S, st, stride = case["batch"], case["frames"], case["blocks"], case["stack"], case["stride"]
    if st > 1 or stride > 1:
        at = (torch.arange(0, T, stride, device=DEV)[:, None] + torch.arange(st, device=DEV)[None, :]).clamp(max=T - 1)
        x = x[:, at].reshape(B, at.shape[0], st * case["dim"])
        T = at.shape[0]
    parts = iter(parts)
    seq, hf, cf = x.double(), [], []
    for l in range(L):
        wx, wh, b = next(parts), next(parts), next(parts).double()
        wp = next(parts) if P > 0 else None
        (ax, Qx), (ah, Qh) = _weights(wx.reshape(4 * H, -1), 4 * S), _weights(wh.reshape(4 * H, -1), 4 * S)
        if P > 0:
            ap, Qp = _weights(wp, S)
        h = h0[l].double() if h0 is not None else torch.zeros((B, R), device=DEV, dtype=torch.float64)
        c = c0[l].double() if c0 is not None else torch.zeros((B, H), device=DEV, dtype=torch.float64)
        out = torch.empty((T, B, R), device=DEV, dtype=torch.float64)
        for t in range(T):
            pre = _layer(seq[:, t], ax, Qx) + b.reshape(-1) + _layer(h, ah, Qh)
            i, f, g, o = pre.reshape(B, 4, H).unbind(1)
            c = torch.sigmoid(f) * c + torch.sigmoid(i) * torch.tanh(g)
            h = torch.sigmoid(o) * torch.tanh(c)
            if P > 0:
                h = _layer(h, ap, Qp)
            out[t] = h
        seq = out.transpose(0, 1)
        hf.append(h)
        cf.append(c)
    y = seq
    if C > 0:
        wo, bo = next(parts), next(parts).double()
        flat = seq.reshape(B * T, R)
        y = torch.empty((B * T, C), device=DEV, dtype=torch.float64)
        w, Qw = (wo.double(), None) if case["mode"] == "float" else _weights(wo, S)
        for r in range(0, B * T, 16384):
            rows = flat[r:r + 16384]
            z = (rows @ w.t() if Qw is None else _layer(rows, w, Qw)) + bo
            y[r:r + 16384] = torch.softmax(z, 1)
        y = y.reshape(B, T, C)
    keep = h0 is not None
    return {"y": y, "h": torch.stack(hf) if keep else None, "c": torch.stack(cf) if keep else None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "quantize":
        return None  # whole numbers
    if kind == "qmatmul":
        w, a, b = _qmatmul_input(case, seed)
        aw, Qw = _weights(w, case["blocks"])
        aa, Qa = _offset_codes(a, 1) if case["per_row"] else _offset_codes(a.reshape(1, -1), 1)
        y = (aa.reshape(case["m"], case["k"]) @ aw.t()) / (Qa * Qw)
        return (y + b.double() if b is not None else y, None)
    if kind == "lstm":
        return _lstm_exact(case, seed)
    g = _gen(seed)
    w = _uniform(g, case["n"], case["k"], a=case["k"] ** -0.5)
    b = _uniform(g, case["n"], a=0.1) if case["bias"] else None
    x = torch.sigmoid(_normal(g, case["m"], case["k"], std=2.0))
    gy = _normal(g, case["m"], case["n"], std=1e-3).double()
    aw, Qw = _weights(w, 1)
    y = _layer(x, aw, Qw)
    return {"y": y + b.double() if b is not None else y, "gx": gy @ w.double(), "gw": gy.t() @ x.double(),
            "gb": gy.sum(0) if b is not None else None}
