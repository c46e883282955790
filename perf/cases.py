"""The calls this library is timed on, and more of the same ranges (`draw`).

A case is one call of a public entry point on rows x cols of one type, with the plan left to the library (the
committed calibration and learned model loaded, as a program that uses the library does at start-up):

  fwd     credit.run_ex: softmax, log-sum-exp, LayerNorm (gamma, beta), RMSNorm (gamma), row-wise int8
          quantisation, in FP32, BF16 and FP8-E4M3 with per-row scales, and the norms quantised to FP8
  bwd     credit.run_bwd: the gradients of softmax, LayerNorm, RMSNorm, of softmax and cross entropy from logits,
          of the weighted variance and of the Pearson correlation
  ragged  one replay of a credit.Ragged batch (softmax / RMSNorm rows of log-uniform width)

Ranges: 64 to 65536 rows of 1K to 1M columns, even, odd and power-of-two widths, up to 4 GiB of inputs and outputs.
"""
import math
import os
import random

import torch

from paper_2609_01864_gb300 import credit as C

DT = {"f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.float8_e4m3fn, "int8": torch.int8}
SIZE = {"f32": 4, "bf16": 2, "fp8": 1, "int8": 1}
CODE = {"f32": C.F32, "bf16": C.BF16, "fp8": C.FP8_E4M3, "int8": C.INT8}
FWD = {"softmax": C.SOFTMAX, "logsumexp": C.LOGSUMEXP, "layernorm": C.LAYERNORM, "rmsnorm": C.RMSNORM,
       "quant_int8": C.QUANT_INT8}
BWD = {"softmax_bwd": C.SOFTMAX_BWD, "layernorm_bwd": C.LAYERNORM_BWD, "rmsnorm_bwd": C.RMSNORM_BWD,
       "softmax_logits_bwd": C.SOFTMAX_LOGITS_BWD, "xent_bwd": C.XENT_BWD, "wvar_bwd": C.WVAR_BWD,
       "pearson_bwd": C.PEARSON_BWD}
PAIR = ("wvar_bwd", "pearson_bwd")
NORMS = ("layernorm", "rmsnorm")
CAP_BYTES = 4 << 30  # inputs and outputs of a drawn case
EXACT_BLOCK = 1 << 26  # elements worked on at once in 64 bits


def _fwd(name, op, dtype, rows, cols, out=None):
    return {"name": name, "kind": "fwd", "op": op, "dtype": dtype, "out": out or dtype, "rows": rows, "cols": cols}


def _bwd(name, op, dtype, rows, cols):
    return {"name": name, "kind": "bwd", "op": op, "dtype": dtype, "rows": rows, "cols": cols}


def listed():
    return [
        # the smallest call: attention-sized rows of a small batch, where the launch and the host path count
        _fwd("softmax_f32_256x4096", "softmax", "f32", 256, 4096),
        # the norm of a hidden state: many rows of a few thousand columns, in the type models run in
        _fwd("rmsnorm_bf16_16384x4096", "rmsnorm", "bf16", 16384, 4096),
        # the same norm handing FP8 codes and row scales to a quantised matrix product
        _fwd("rmsnorm_bf16_fp8_16384x8192", "rmsnorm", "bf16", 16384, 8192, out="fp8"),
        # a width that no vector length divides: every row starts at another offset
        _fwd("layernorm_bf16_4096x30001", "layernorm", "bf16", 4096, 30001),
        # the widest rows of the FP32 norm workload (the largest single call)
        _fwd("layernorm_f32_4096x262144", "layernorm", "f32", 4096, 262144),
        # few, very wide rows: less than a row per SM
        _fwd("rmsnorm_f32_64x1048576", "rmsnorm", "f32", 64, 1048576),
        # logits over a vocabulary in BF16 and in FP8, and their log-sum-exp at an odd vocabulary size
        _fwd("softmax_bf16_4096x131072", "softmax", "bf16", 4096, 131072),
        _fwd("softmax_fp8_4096x131072", "softmax", "fp8", 4096, 131072),
        _fwd("logsumexp_bf16_8192x32003", "logsumexp", "bf16", 8192, 32003, out="f32"),
        # a training step's backward passes: the norm of the hidden state, the loss over the vocabulary
        _bwd("layernorm_bwd_bf16_16384x4096", "layernorm_bwd", "bf16", 16384, 4096),
        _bwd("xent_bwd_bf16_4096x131072", "xent_bwd", "bf16", 4096, 131072),
        # a packed batch of rows of uneven width and mixed op
        {"name": "ragged_bf16_20000", "kind": "ragged", "dtype": "bf16", "rows": 20000, "lo": 1024, "hi": 1048576},
    ]


def _bytes(kind, op, dtype, out, rows, cols):
    n, i = rows * cols, SIZE[dtype]
    if kind == "bwd":
        return n * i * (4 if op in PAIR else 3)
    return n * i + (rows * 4 if op == "logsumexp" else n * SIZE[out])


def draw(rng):
    kind = rng.choice(("fwd",) * 6 + ("bwd",) * 3 + ("ragged",))
    if kind == "ragged":
        lo = int(round(2 ** rng.uniform(10, 14)))
        return {"kind": "ragged", "dtype": rng.choice(("bf16", "f32")), "rows": int(round(2 ** rng.uniform(6, 12))),
                "lo": lo, "hi": int(round(lo * 2 ** rng.uniform(1, 5)))}
    if kind == "bwd":
        op, dtype = rng.choice(sorted(BWD)), rng.choice(("f32", "bf16"))
        out = dtype
    else:
        op = rng.choice(("softmax", "logsumexp", "layernorm", "rmsnorm", "layernorm", "rmsnorm", "quant_int8"))
        dtype = rng.choice(("f32", "bf16") if op == "quant_int8" else ("f32", "bf16", "fp8"))
        out = "f32" if op == "logsumexp" else "int8" if op == "quant_int8" else dtype
        if op in NORMS and dtype == "bf16" and rng.random() < 0.25:
            out = "fp8"
    while True:
        rows, cols = int(round(2 ** rng.uniform(6, 16))), int(round(2 ** rng.uniform(10, 20)))
        form = rng.choice(("any", "sixteen", "power"))
        if form == "sixteen":
            cols = cols // 16 * 16
        elif form == "power":
            cols = 1 << int(round(math.log2(cols)))
        if _bytes(kind, op, dtype, out, rows, cols) <= CAP_BYTES:
            break
    c = {"kind": kind, "op": op, "dtype": dtype, "rows": rows, "cols": cols}
    if kind == "fwd":
        c["out"] = out
    return c


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(g, rows, cols, std, dtype):
    x = torch.randn(rows, cols, generator=g, device="cuda", dtype=DT[dtype] if dtype == "bf16" else torch.float32)
    return x if std == 1.0 else x.mul_(std)


def _activations(g, rows, cols, dtype):
    """N(0, 1) with 1% of the elements at +-50."""
    x = _normal(g, rows, cols, 1.0, dtype)
    step = max(1, EXACT_BLOCK // cols)
    for r in range(0, rows, step):
        v = x[r:r + step]
        u = torch.rand(v.shape, generator=g, device="cuda")
        v.masked_fill_(u < 0.005, 50.0).masked_fill_(u > 0.995, -50.0)
    return x


def _e4m3(x):
    """FP8 codes and per-row scales amax / 448."""
    q = torch.empty(x.shape, device="cuda", dtype=torch.float8_e4m3fn)
    s = torch.empty(x.shape[0], device="cuda")
    step = max(1, EXACT_BLOCK // x.shape[1])
    for r in range(0, x.shape[0], step):
        v = x[r:r + step]
        s[r:r + step] = v.abs().amax(1) / 448.0
        q[r:r + step] = (v / s[r:r + step, None]).clamp_(-448, 448).to(torch.float8_e4m3fn)
    return q, s


def _inputs(case, seed):
    g = _gen(seed)
    dtype, rows = case["dtype"], case["rows"]
    if case["kind"] == "ragged":
        shape = random.Random(rows + case["lo"] + case["hi"])  # the widths and ops belong to the case
        span = math.log2(case["hi"] / case["lo"])
        widths = [int(round(case["lo"] * 2 ** (span * shape.random()))) for _ in range(rows)]
        ops = [shape.random() < 0.5 for _ in range(rows)]
        off, table = 0, []
        for w, o in zip(widths, ops):
            table.append((off, off, w, C.SOFTMAX if o else C.RMSNORM))
            off += w
        return {"x": _normal(g, 1, off, 1.0, dtype)[0], "rows": table}
    op, cols = case["op"], case["cols"]
    gamma = 1.0 + 0.1 * torch.randn(cols, generator=g, device="cuda")
    beta = 0.1 * torch.randn(cols, generator=g, device="cuda")
    if case["kind"] == "fwd":
        x = (_normal(g, rows, cols, 3.0, dtype) if op in ("softmax", "logsumexp") else _activations(g, rows, cols, dtype))
        d = {"x": x}
        if dtype == "fp8":
            d["x"], d["in_scale"] = _e4m3(x)
        if op in NORMS:
            d["gamma"] = gamma
        if op == "layernorm":
            d["beta"] = beta
        return d
    d = {}
    if op in ("layernorm_bwd", "rmsnorm_bwd"):
        a = _activations(g, rows, cols, dtype)
        step = max(1, EXACT_BLOCK // cols)
        mean, rstd = torch.empty(rows, device="cuda"), torch.empty(rows, device="cuda")
        for r in range(0, rows, step):  # the row statistics that the forward saved
            v = a[r:r + step].double()
            if op == "layernorm_bwd":
                mean[r:r + step] = v.mean(1)
                rstd[r:r + step] = (v.var(1, correction=0) + 1e-5).rsqrt()
            else:
                rstd[r:r + step] = (v.square().mean(1) + 1e-6).rsqrt()
        d.update(gamma=gamma, rstd=rstd)
        if op == "layernorm_bwd":
            d["mean"] = mean
    elif op == "softmax_bwd":
        a = torch.softmax(_normal(g, rows, cols, 3.0, dtype), 1)
    elif op in ("softmax_logits_bwd", "xent_bwd"):
        a = _normal(g, rows, cols, 3.0, dtype)
    else:
        a = _normal(g, rows, cols, 1.0, dtype)
    if op == "xent_bwd":  # soft targets
        dy = torch.softmax(_normal(g, rows, cols, 2.0, dtype), 1)
    elif op == "wvar_bwd":  # weights
        dy = torch.rand(rows, cols, generator=g, device="cuda", dtype=DT[dtype])
    elif op == "pearson_bwd":  # a second variable, correlated with the first
        dy = _normal(g, rows, cols, 1.0, dtype).add_(a, alpha=0.5)
    else:
        dy = _normal(g, rows, cols, 1.0, dtype)
    if op in PAIR or op == "xent_bwd":
        d["scale"] = 0.5 + torch.rand(rows, generator=g, device="cuda")
    return {"a": a, "dy": dy, "kw": d}


# ---------------------------------------------------------------- the calls
_ready = False


def _start():
    """What a program does once: bring the device up and load the committed calibration and learned model."""
    global _ready
    if not _ready:
        C.init()
        C.load_model(os.path.join(os.path.dirname(C.__file__), "data", "gb300.calib"))
        _ready = True


def prepare(case, seed):
    _start()
    d = _inputs(case, seed)
    rows = case["rows"]
    if case["kind"] == "ragged":
        y = torch.empty_like(d["x"])
        torch.cuda.synchronize()  # the batch is timed on its inputs when the handle is made
        return {"kind": "ragged", "x": d["x"], "y": y, "h": C.Ragged(d["rows"], CODE[case["dtype"]], d["x"], y)}
    if case["kind"] == "bwd":
        kw = d["kw"]
        s = {"kind": "bwd", "op": BWD[case["op"]], "a": d["a"], "dy": d["dy"], "dx": torch.empty_like(d["a"])}
        if case["op"] in PAIR:
            kw["dx2"] = torch.empty_like(d["a"])
        s["kw"] = kw
        return s
    op = case["op"]
    y = torch.empty((rows,) if op == "logsumexp" else (rows, case["cols"]), device="cuda", dtype=DT[case["out"]])
    kw = dict(in_dtype=CODE[case["dtype"]], out_dtype=CODE[case["out"]], in_scale=d.get("in_scale"),
              gamma=d.get("gamma"), beta=d.get("beta"))
    if case["out"] in ("fp8", "int8"):
        kw["out_scale"] = torch.empty(rows, device="cuda")
    return {"kind": "fwd", "op": FWD[op], "x": d["x"], "y": y, "kw": kw}


def run(state):
    if state["kind"] == "ragged":
        state["h"].run()
        return state["y"]
    kw = state["kw"]
    if state["kind"] == "bwd":
        C.run_bwd(state["op"], state["a"], state["dy"], state["dx"], **kw)
        return [state["dx"], kw["dx2"]] if "dx2" in kw else state["dx"]
    C.run_ex(state["op"], state["x"], state["y"], **kw)
    return [state["y"], kw["out_scale"]] if "out_scale" in kw else state["y"]


def work(case):
    if case["kind"] == "ragged":
        # rows times the mean of a log-uniform width
        n = case["rows"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return {"bytes": 2 * n * SIZE[case["dtype"]], "flops": 4 * n}
    n = case["rows"] * case["cols"]
    return {"bytes": _bytes(case["kind"], case["op"], case["dtype"], case.get("out"), case["rows"], case["cols"]),
            "flops": (10 if case["kind"] == "bwd" else 5) * n}


# ---------------------------------------------------------------- the results in 64 bits
def _exact_fwd(op, x, d, quant):
    """(result, amax of the result's row where it is handed on as FP8 codes)."""
    if op == "logsumexp":
        return torch.logsumexp(x, 1), None
    if op == "softmax":
        y = torch.softmax(x, 1)
    else:
        if op == "layernorm":
            x = x - x.mean(1, keepdim=True)
        y = x * (x.square().mean(1, keepdim=True) + (1e-5 if op == "layernorm" else 1e-6)).rsqrt() * d["gamma"].double()
        if op == "layernorm":
            y += d["beta"].double()
    return y, (y.abs().amax(1) if quant else None)


def _exact_bwd(op, a, dy, kw):
    n = a.shape[1]
    col = {k: v[:, None] for k, v in kw.items() if k != "gamma"}
    if op == "softmax_bwd":
        return [a * (dy - (a * dy).sum(1, keepdim=True))]
    if op in ("softmax_logits_bwd", "xent_bwd"):
        y = torch.softmax(a, 1)
        if op == "xent_bwd":
            return [col["scale"] * (y * dy.sum(1, keepdim=True) - dy)]
        return [y * (dy - (y * dy).sum(1, keepdim=True))]
    if op in ("layernorm_bwd", "rmsnorm_bwd"):
        xh = (a - col["mean"] if op == "layernorm_bwd" else a) * col["rstd"]
        g = dy * kw["gamma"]
        dx = g - xh * ((g * xh).sum(1, keepdim=True) / n)
        if op == "layernorm_bwd":
            dx -= g.mean(1, keepdim=True)
        return [dx * col["rstd"]]
    if op == "wvar_bwd":
        w = dy.sum(1, keepdim=True)
        u = a - (dy * a).sum(1, keepdim=True) / w
        v = (dy * u * u).sum(1, keepdim=True) / w
        return [col["scale"] * 2 * dy * u / w, col["scale"] * (u * u - v) / w]
    u, v = a - a.mean(1, keepdim=True), dy - dy.mean(1, keepdim=True)
    sxx, syy, sxy = u.square().sum(1, keepdim=True), v.square().sum(1, keepdim=True), (u * v).sum(1, keepdim=True)
    den = (sxx * syy).sqrt()
    r = sxy / den
    return [col["scale"] * (v / den - r * u / sxx), col["scale"] * (u / den - r * v / syy)]


def exact(case, seed):
    d = _inputs(case, seed)
    rows = case["rows"]
    if case["kind"] == "ragged":
        y = torch.empty(d["x"].shape, device="cuda", dtype=torch.float64)
        for i, _, w, op in d["rows"]:
            x = d["x"][i:i + w].double()
            y[i:i + w] = torch.softmax(x, 0) if op == C.SOFTMAX else x * (x.square().mean() + 1e-6).rsqrt()
        return y
    op, cols = case["op"], case["cols"]
    step = max(1, EXACT_BLOCK // cols)
    parts = []
    for r in range(0, rows, step):
        if case["kind"] == "bwd":
            kw = {k: (v if k == "gamma" else v[r:r + step]).double() for k, v in d["kw"].items()}
            parts.append(_exact_bwd(op, d["a"][r:r + step].double(), d["dy"][r:r + step].double(), kw))
            continue
        x = d["x"][r:r + step].double()
        if "in_scale" in d:
            x *= d["in_scale"][r:r + step, None].double()
        if op == "quant_int8":
            parts.append((None, x.abs().amax(1) / 127))
            continue
        y, amax = _exact_fwd(op, x, d, case["out"] == "fp8")
        if amax is None:
            parts.append((y,))
        else:  # the values that the codes stand for, before they are rounded to FP8
            parts.append((y.mul_((448 / amax)[:, None]), amax / 448))
    out = [None if v[0] is None else torch.cat(v) for v in zip(*parts)]
    return out[0] if len(out) == 1 else out
