"""The work that users of this library have it do, as cases that can be timed.

Three kinds of program use it: a QAT trainer (fake-quant of weights and activations in every step), a
checkpoint writer (anchor quantization of a whole weight set, once per checkpoint) and a server that
lowers a stored anchor to the precision it needs (one tensor, one decoder layer or the whole model at a
time) and reconstructs or hands the result to a block-scaled matrix multiply.  Shapes are those of the
8B Llama-shaped weight set of `inputs.LLAMA8B_LAYER`, of the two single-matrix workloads of the bench
(FP32 4096 x 4096, BF16 8192 x 8192), of its [8, 4096, 4096] activations, and a decoded token, a chat
turn or a prefill of the same width.

A case names a path, its formats and its sizes; `run` goes through the package's public entry points.
Every result is defined bit for bit, so all comparisons are exact.
"""
from __future__ import annotations

import math

import torch

import paper_2604_00529_b200 as mxq
from paper_2604_00529_b200 import inputs

BITS = {"int8": 8, "int7": 7, "int6": 6, "int5": 5, "int4": 4, "int3": 3, "int2": 2,
        "e4m3": 8, "e3m3": 7, "e3m2": 6, "e2m3": 6, "e2m2": 5, "e2m1": 4}
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
MODES = {"direct": mxq.FQ_DIRECT, "via_anchor": mxq.FQ_VIA_ANCHOR}


def listed():
    return [
        # one decoded token's activations on their way into a block-scaled matmul: the smallest call there is
        {"name": "token_quantize", "path": "quantize", "rows": 1, "cols": 4096, "dtype": "bf16", "values": "activations",
         "fmt": "e4m3", "block": 32},
        # the activations of one training chat turn inside the autograd graph of a QAT step, forward and backward
        {"name": "ste_chat_turn", "path": "ste", "rows": 512, "cols": 4096, "dtype": "bf16", "values": "activations",
         "fmt": "e2m1", "block": 32, "mode": "via_anchor", "copy_grad": False},
        # a server lowers one small projection just before it is used: buffers persist, calls are prepared once
        {"name": "projection_on_demand", "path": "on_demand", "rows": 1024, "cols": 4096, "dtype": "bf16",
         "values": "weights", "src": "int8", "fmt": "int4", "block": 32},
        # a prefill of 1000 tokens quantized for a block-scaled matmul: rows do not fill the last scale tile
        {"name": "prefill_tiled", "path": "quantize_tiled", "rows": 1000, "cols": 4096, "dtype": "bf16",
         "values": "activations", "fmt": "e4m3", "block": 32},
        # the FP32 master matrix of the first bench workload: anchor, lower format, reconstruction
        {"name": "master_f32_chain", "path": "chain", "rows": 4096, "cols": 4096, "dtype": "f32", "values": "weights",
         "src": "int8", "fmt": "int4", "block": 32},
        # one heavy-tailed BF16 matrix (second bench workload) served in two lower precisions from one anchor
        {"name": "elastic_two_targets", "path": "multi", "rows": 8192, "cols": 8192, "dtype": "bf16", "values": "heavy",
         "src": "e4m3", "fmts": "e2m3,e2m1", "block": 32},
        # the widths a multi-format model is evaluated at without having been trained on them, at the block size
        # of the paper's tensor-level study, from one MLP weight
        {"name": "unseen_widths", "path": "multi", "rows": 14336, "cols": 4096, "dtype": "bf16", "values": "weights",
         "src": "int8", "fmts": "int7,int5,int3", "block": 64},
        # the seven linear weights of one decoder layer lowered and reconstructed by the two batched launches
        {"name": "layer_lower_reconstruct", "path": "set_lower", "layers": 1, "hidden": 4096, "kv": 1024, "mlp": 14336,
         "dtype": "bf16", "values": "weights", "src": "e4m3", "fmt": "e2m3", "block": 32},
        # the activations of a training batch, fake-quant forward and straight-through backward
        {"name": "batch_activations", "path": "fake_quant", "rows": 8 * 4096, "cols": 4096, "dtype": "bf16",
         "values": "activations", "fmt": "int6", "block": 32, "mode": "via_anchor"},
        # the FP32 master weights of four layers of a QAT step in one launch
        {"name": "qat_weights_f32", "path": "set_fake_quant", "layers": 4, "hidden": 4096, "kv": 1024, "mlp": 14336,
         "dtype": "f32", "values": "weights", "fmt": "int4", "block": 32, "mode": "via_anchor"},
        # a quarter of the model into its MXINT8 anchor checkpoint
        {"name": "anchor_checkpoint", "path": "set_quantize", "layers": 8, "hidden": 4096, "kv": 1024, "mlp": 14336,
         "dtype": "bf16", "values": "weights", "fmt": "int8", "block": 32},
        # the whole model's stored anchors into the two precisions it is served in
        {"name": "model_two_precisions", "path": "set_pair", "layers": 32, "hidden": 4096, "kv": 1024, "mlp": 14336,
         "dtype": "bf16", "values": "weights", "src": "e4m3", "fmts": "e2m3,e2m1", "block": 32},
    ]


# ---- drawn cases -----------------------------------------------------------------------------

INT_TARGETS = ("int6", "int4", "int7", "int5", "int3", "int2")
FP_TARGETS = ("e2m3", "e2m1", "e3m2", "e3m3", "e2m2")
PATHS = ("quantize", "ste", "on_demand", "quantize_tiled", "lower_tiled", "chain", "multi", "lower", "reconstruct",
         "fake_quant", "set_lower", "set_fake_quant", "set_quantize", "set_pair")


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(PATHS)
    integer = rng.random() < 0.5 and "tiled" not in path
    src = "int8" if integer else "e4m3"
    # the formats of the workloads more often than the other ones
    targets = INT_TARGETS if integer else FP_TARGETS
    fmt = rng.choice(targets[:3] if rng.random() < 0.6 else targets)
    case = {"path": path, "dtype": rng.choice(("bf16", "bf16", "f32"))}
    block = 32 if "tiled" in path or rng.random() < 0.6 else rng.choice((16, 64, 128))
    if path in ("multi", "set_lower", "set_pair") or path.startswith("set_"):
        block = max(block, 32)
    case["block"] = block
    if path.startswith("set_"):
        unit = 128
        case.update(layers=_log_int(rng, 1, 8), hidden=unit * _log_int(rng, 2, 32), kv=unit * _log_int(rng, 1, 8),
                    mlp=unit * _log_int(rng, 4, 112), values="weights")
    else:
        # rows of any number, columns of any whole number of blocks (and of 32, which packed codes need)
        step = max(block, 32)
        total = math.exp(rng.uniform(math.log(4096), math.log(1 << 27)))
        cols = step * max(1, _log_int(rng, 256, 14336) // step)
        case.update(rows=max(1, int(total / cols)), cols=cols,
                    values=rng.choice(("weights", "heavy", "activations")))
    if path in ("quantize", "set_quantize"):
        case["fmt"] = src if rng.random() < 0.5 else fmt
    elif path == "quantize_tiled":
        case["fmt"] = rng.choice(("e4m3", "e2m3", "e3m2", "e2m1"))
    elif path == "lower_tiled":
        case.update(src=src, fmt=rng.choice(("e2m3", "e3m2", "e2m1")))
    elif path in ("ste", "fake_quant", "set_fake_quant"):
        case.update(fmt=src if rng.random() < 0.2 else fmt, mode=rng.choice(("direct", "via_anchor", "via_anchor")))
        if path == "ste":
            case["copy_grad"] = rng.random() < 0.3
    elif path in ("multi", "set_pair"):
        count = 2 if path == "set_pair" else rng.choice((2, 2, 3, 4))
        case.update(src=src, fmts=",".join(rng.sample(targets, count)))
    elif path == "lower":
        # mostly from the anchor; sometimes a server that kept only a 6-bit set goes down to four bits
        if rng.random() < 0.25:
            case.update(src="int6" if integer else rng.choice(("e3m2", "e2m3")), fmt="int4" if integer else "e2m1")
        else:
            case.update(src=src, fmt=fmt)
    elif path == "reconstruct":
        case["fmt"] = src if rng.random() < 0.4 else fmt
    else:                                       # chain, on_demand, set_lower
        case.update(src=src, fmt=fmt)
    return case


# ---- inputs ----------------------------------------------------------------------------------

def _tensor(gen, rows, cols, dtype, values):
    """rows x cols values of the kind the path meets: weights N(0, 0.02^2); heavy-tailed weights (a ratio of
    normals cut at 8 deviations, with 0.1 % outliers x 50); activations N(0, 1) with 1 % hot channels x 20."""
    dt = DTYPES[dtype]
    x = torch.randn(rows, cols, device="cuda", dtype=dt, generator=gen)
    if values == "activations":
        hot = torch.randperm(cols, device="cuda", generator=gen)[:max(1, cols // 100)]
        x[:, hot] *= 20
    elif values == "heavy":
        x /= torch.randn(rows, cols, device="cuda", dtype=dt, generator=gen).abs_().add_(0.25)
        x.clamp_(-8, 8).mul_(0.02)
        x[torch.rand(rows, cols, device="cuda", generator=gen) < 0.001] *= 50
    else:
        x *= 0.02
    return x


def _shapes(case):
    """The linear weights of the case's decoder layers, in the order of `inputs.LLAMA8B_LAYER`."""
    rows = {"q": case["hidden"], "o": case["hidden"], "k": case["kv"], "v": case["kv"],
            "gate": case["mlp"], "up": case["mlp"], "down": case["hidden"]}
    one = [(rows[name], case["mlp"] if name == "down" else case["hidden"]) for name, _, _ in inputs.LLAMA8B_LAYER]
    return one * case["layers"]


class _Arena:
    """One allocation cut into the pieces of a weight set (every piece starts on a 256-byte boundary)."""

    def __init__(self, sizes, dtype=torch.uint8):
        item = torch.empty(0, dtype=dtype).element_size()
        at, where = 0, []
        for n in sizes:
            where.append((at, at + n))
            at += -(-n * item // 256) * 256 // item
        self.whole = torch.zeros(at, dtype=dtype, device="cuda")
        self.parts = [self.whole[a:b] for a, b in where]


def _codes(case_fmts, sizes):
    return [_Arena([n * BITS[f] // 8 for n in sizes]) for f in case_fmts]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    path, block = case["path"], case["block"]
    s = {"case": case}
    if path.startswith("set_"):
        return _prepare_set(case, s, gen)
    rows, cols = case["rows"], case["cols"]
    n = s["n"] = rows * cols
    x = _tensor(gen, rows, cols, case["dtype"], case["values"])
    if path in ("quantize", "quantize_tiled", "chain"):
        s["x"] = x
    elif path == "ste":
        s["x"] = x.requires_grad_()
        s["grad"] = torch.randn(rows, cols, device="cuda", dtype=x.dtype, generator=gen)
    elif path == "fake_quant":
        s["x"] = x
        s["grad"] = torch.randn(rows, cols, device="cuda", dtype=x.dtype, generator=gen)
    elif path == "reconstruct":
        s["codes"], s["scales"] = mxq.quantize(x, case["fmt"], block)
    else:                                       # lower, lower_tiled, multi, on_demand: a stored anchor
        s["codes"], s["scales"] = mxq.quantize(x, case["src"], block)
    if path == "on_demand":
        fmt = case["fmt"]
        low = torch.empty(mxq.codes_bytes(n, fmt), dtype=torch.uint8, device="cuda")
        low_scales = torch.empty(n // block, dtype=torch.uint8, device="cuda")
        out = torch.empty(rows, cols, dtype=DTYPES[case["dtype"]], device="cuda")
        s["lower"] = mxq.prepare_slice_scale(s["codes"], s["scales"], n, case["src"], fmt, block, low, low_scales)
        s["reconstruct"] = mxq.prepare_dequantize(low, low_scales, n, fmt, block, out)
        s["out"] = (low, low_scales, out)
    return s


def _prepare_set(case, s, gen):
    path, block, dtype = case["path"], case["block"], case["dtype"]
    shapes = _shapes(case)
    sizes = [r * c for r, c in shapes]
    scales = [n // block for n in sizes]
    if path in ("set_quantize", "set_fake_quant"):
        src = _Arena(sizes, DTYPES[dtype])
        for part, (r, c) in zip(src.parts, shapes):
            part.copy_(_tensor(gen, r, c, dtype, case["values"]).view(-1))
        if path == "set_quantize":
            codes, sc = _Arena([n * BITS[case["fmt"]] // 8 for n in sizes]), _Arena(scales)
            s["table"] = mxq.make_q_items(list(zip(src.parts, codes.parts, sc.parts)))
            s["out"] = (codes.whole, sc.whole)
        else:
            dst = _Arena(sizes, DTYPES[dtype])
            s["table"] = mxq.make_fq_items(list(zip(src.parts, dst.parts)))
            s["out"] = (dst.whole,)
        return s
    anchor, anchor_scales = _Arena(sizes), _Arena(scales)
    for c, sc, (rows, cols) in zip(anchor.parts, anchor_scales.parts, shapes):
        mxq.quantize(_tensor(gen, rows, cols, dtype, case["values"]), case["src"], block, c, sc)
    fmts = case["fmts"].split(",") if path == "set_pair" else [case["fmt"]]
    low = _codes(fmts, sizes)
    low_scales = [_Arena(scales) for _ in fmts]
    if path == "set_pair":
        s["table"] = mxq.make_pair_items(list(zip(anchor.parts, anchor_scales.parts, sizes, low[0].parts, low_scales[0].parts,
                                                  low[1].parts, low_scales[1].parts)))
        s["out"] = (low[0].whole, low_scales[0].whole, low[1].whole, low_scales[1].whole)
    else:
        dst = _Arena(sizes, DTYPES[dtype])
        s["table"] = mxq.make_items(list(zip(anchor.parts, anchor_scales.parts, sizes, low[0].parts, low_scales[0].parts)))
        s["back"] = mxq.make_dq_items(list(zip(low[0].parts, low_scales[0].parts, sizes, dst.parts)))
        s["out"] = (low[0].whole, low_scales[0].whole, dst.whole)
    return s


# ---- one pass --------------------------------------------------------------------------------

def run(s):
    case = s["case"]
    path, block = case["path"], case["block"]
    if path == "quantize":
        return mxq.quantize(s["x"], case["fmt"], block)
    if path == "ste":
        y = mxq.fake_quant_ste(s["x"], case["fmt"], block, MODES[case["mode"]], case["copy_grad"])
        (g,) = torch.autograd.grad(y, s["x"], s["grad"])
        return y, g
    if path == "on_demand":
        s["lower"]()
        s["reconstruct"]()
        return s["out"]
    if path == "quantize_tiled":
        return mxq.quantize_tiled(s["x"], case["fmt"])
    if path == "lower_tiled":
        return mxq.slice_scale_tiled(s["codes"], s["scales"], case["rows"], case["cols"], case["src"], case["fmt"])
    if path == "chain":
        codes, scales = mxq.quantize(s["x"], case["src"], block)
        low, low_scales = mxq.slice_scale(codes, scales, s["n"], case["src"], case["fmt"], block)
        back = mxq.dequantize(low, low_scales, s["n"], case["fmt"], block, dtype=DTYPES[case["dtype"]])
        return codes, scales, low, low_scales, back
    if path == "multi":
        return mxq.slice_scale_multi(s["codes"], s["scales"], s["n"], case["src"], case["fmts"].split(","), block)
    if path == "lower":
        return mxq.slice_scale(s["codes"], s["scales"], s["n"], case["src"], case["fmt"], block)
    if path == "reconstruct":
        return mxq.dequantize(s["codes"], s["scales"], s["n"], case["fmt"], block, dtype=DTYPES[case["dtype"]])
    if path == "fake_quant":
        return mxq.fake_quant(s["x"], case["fmt"], block, MODES[case["mode"]]), mxq.fake_quant_bwd(s["grad"])
    if path == "set_quantize":
        mxq.quantize_batched(s["table"], case["fmt"], block)
    elif path == "set_fake_quant":
        mxq.fake_quant_batched(s["table"], case["fmt"], block, MODES[case["mode"]])
    elif path == "set_pair":
        first, second = case["fmts"].split(",")
        mxq.slice_scale_pair_batched(s["table"], case["src"], first, second, block)
    else:
        mxq.slice_scale_batched(s["table"], case["src"], case["fmt"], block)
        mxq.dequantize_batched(s["back"], case["fmt"], block)
    return s["out"]


# ---- what a pass cannot do without ------------------------------------------------------------

def work(case):
    """Bytes of the pass: every input read once, every output written once (the library does a few integer
    or conversion operations per element and no arithmetic that a FLOP rate would bound)."""
    path, block = case["path"], case["block"]
    n = sum(r * c for r, c in _shapes(case)) if path.startswith("set_") else case["rows"] * case["cols"]
    size = 4 if case["dtype"] == "f32" else 2
    scale = 1 / block

    def stored(fmt):
        return BITS[fmt] / 8 + scale

    if path in ("quantize", "quantize_tiled", "set_quantize"):
        per = size + stored(case["fmt"])
    elif path == "ste":
        per = 2 * size + (2 * size if case["copy_grad"] else 0)
    elif path == "fake_quant":
        per = 4 * size
    elif path == "set_fake_quant":
        per = 2 * size
    elif path in ("multi", "set_pair"):
        per = stored(case["src"]) + sum(stored(f) for f in case["fmts"].split(","))
    elif path in ("lower", "lower_tiled"):
        per = stored(case["src"]) + stored(case["fmt"])
    elif path == "reconstruct":
        per = stored(case["fmt"]) + size
    elif path in ("on_demand", "set_lower"):
        per = stored(case["src"]) + stored(case["fmt"]) + size        # the lower codes are a result that is kept
    else:                                                             # chain: both code sets are results
        per = size + stored(case["src"]) + stored(case["fmt"]) + size
    return {"bytes": float(n * per), "flops": 0.0}


def tolerance(case):
    return "exact"
