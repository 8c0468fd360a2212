"""The work whose speed is measured: products as programs call them.

Every case names a `path` (the entry point and mode), its sizes and the values
its inputs take:

  gemm     C = A.B, one product queued on the caller's stream (mm_gemm_async)
  axpby    C = alpha A.B + beta D (mm_gemm_axpby_async)
  grouped  many independent products in one call (mm_gemm_grouped_async)
  serve    requests submitted to the serving loop, then waited for
           (mm_submit / mm_wait)

Inputs are on the device, made from a seed.  `listed` gives the fixed cases,
`draw` more of the same ranges.
"""
from __future__ import annotations

import math
import random

import torch

import paper_1306_6192_gb300 as mm

MODES = {
    "auto_f32": (mm.MM_F32, mm.MM_MODE_AUTO),
    "simt": (mm.MM_F32, mm.MM_MODE_SIMT),
    "fp8": (mm.MM_F32, mm.MM_MODE_FP8),
    "auto_f64": (mm.MM_F64, mm.MM_MODE_AUTO),
    "ozaki": (mm.MM_F64, mm.MM_MODE_OZAKI),
}


def _gemm(name, mode, n, m, p, values="uniform"):
    return {"name": name, "path": "gemm", "mode": mode, "n": n, "m": m, "p": p, "values": values}


def listed():
    return [
        # the plain FP32 kernel on a small square: one launch's latency counts
        _gemm("simt_256", "simt", 256, 256, 256),
        # a skinny product (a few rows against a long inner dimension): bandwidth
        _gemm("skinny_64x16384x64", "auto_f32", 64, 16384, 64),
        # an ordinary small square, fewer output tiles than SMs
        _gemm("square_1024", "auto_f32", 1024, 1024, 1024),
        # sizes as data gives them: no multiple of anything, unaligned rows
        _gemm("ragged_1501x1999x1277", "auto_f32", 1501, 1999, 1277, "normal"),
        # a low-rank update of a large matrix: C = A.B - D, short inner dimension
        {"name": "update_8192x512x8192", "path": "axpby", "mode": "auto_f32", "n": 8192, "m": 512,
         "p": 8192, "alpha": 1.0, "beta": -1.0, "values": "uniform"},
        # the large square that throughput is quoted on
        _gemm("square_8192", "auto_f32", 8192, 8192, 8192),
        # entries over forty binades: the scaled split
        _gemm("wide_4096", "auto_f32", 4096, 4096, 4096, "wide"),
        # FP64 by default
        _gemm("f64_1024", "auto_f64", 1024, 1024, 1024),
        # FP64 emulated on the tensor cores
        _gemm("ozaki_4096", "ozaki", 4096, 4096, 4096),
        # e4m3 operands, scales per block
        _gemm("fp8_4096", "fp8", 4096, 4096, 4096),
        # a batch of uneven products in one call
        {"name": "grouped_1024", "path": "grouped", "mode": "auto_f32", "count": 1024, "lo": 32,
         "hi": 1024, "step": 32, "dims_seed": 4, "values": "uniform"},
        # a burst of requests of mixed size and precision through the serving loop
        {"name": "serve_192", "path": "serve", "mode": "auto_f32", "count": 192, "lo": 64,
         "hi": 4096, "f64_share": 0.2, "dims_seed": 5, "values": "normal"},
    ]


def _size(rng, lo, hi):
    """Log-uniform in [lo, hi]; half of the sizes rounded to a multiple of 32."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.5:
        v = max(32, (v + 16) // 32 * 32)
    return max(lo, min(hi, v))


def draw(rng):
    kind = rng.choice(["simt", "skinny", "product", "product", "update", "wide", "f64", "ozaki", "fp8",
                       "grouped", "serve"])
    values = rng.choice(["uniform", "normal"])
    if kind == "simt":
        case = _gemm(None, "simt", _size(rng, 32, 2048), _size(rng, 32, 2048), _size(rng, 32, 2048), values)
    elif kind == "skinny":
        case = _gemm(None, "auto_f32", _size(rng, 16, 128), _size(rng, 2048, 32768), _size(rng, 16, 128),
                     values)
    elif kind == "product":
        case = _gemm(None, "auto_f32", _size(rng, 64, 8192), _size(rng, 64, 8192), _size(rng, 64, 8192),
                     values)
    elif kind == "update":
        case = {"path": "axpby", "mode": "auto_f32", "n": _size(rng, 256, 8192), "m": _size(rng, 64, 2048),
                "p": _size(rng, 256, 8192), "alpha": rng.choice([1.0, -0.5]),
                "beta": rng.choice([1.0, -1.0, 0.75]), "values": values}
    elif kind == "wide":
        case = _gemm(None, "auto_f32", _size(rng, 256, 4096), _size(rng, 256, 8192), _size(rng, 256, 4096),
                     "wide")
    elif kind == "f64":
        case = _gemm(None, "auto_f64", _size(rng, 64, 1536), _size(rng, 64, 1536), _size(rng, 64, 1536),
                     values)
    elif kind == "ozaki":
        case = _gemm(None, "ozaki", _size(rng, 256, 4096), _size(rng, 256, 4096), _size(rng, 256, 4096),
                     values)
    elif kind == "fp8":
        case = _gemm(None, "fp8", _size(rng, 256, 8192), _size(rng, 256, 8192), _size(rng, 256, 8192), values)
    elif kind == "grouped":
        case = {"path": "grouped", "mode": "auto_f32", "count": _size(rng, 32, 1024), "lo": 32, "hi": 1024,
                "step": rng.choice([1, 32]), "dims_seed": rng.randrange(1 << 30), "values": values}
    else:
        case = {"path": "serve", "mode": "auto_f32", "count": _size(rng, 32, 192), "lo": 64, "hi": 4096,
                "f64_share": 0.2, "dims_seed": rng.randrange(1 << 30), "values": values}
    case.pop("name", None)
    return case


def _problems(case):
    """(n, m, p, mode) of every product of a case."""
    if case["path"] in ("gemm", "axpby"):
        return [(case["n"], case["m"], case["p"], case["mode"])]
    rng = random.Random(case["dims_seed"])
    out = []
    for _ in range(case["count"]):
        if case["path"] == "grouped":  # uniform over lo, lo + step, ..., hi
            d = [rng.randrange(case["lo"], case["hi"] + 1, case["step"]) for _ in range(3)]
            out.append((*d, case["mode"]))
        else:  # log-uniform over [lo, hi], a share of FP64 requests
            d = [int(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]))))) for _ in range(3)]
            out.append((*d, "ozaki" if rng.random() < case["f64_share"] else case["mode"]))
    return out


def _values(gen, kind, shape, dtype):
    if kind == "normal":
        return torch.randn(shape, generator=gen, device="cuda", dtype=dtype)
    if kind == "wide":  # sign 2^e, e uniform in [-20, 20)
        e = torch.rand(shape, generator=gen, device="cuda", dtype=dtype) * 40.0 - 20.0
        sign = torch.randint(0, 2, shape, generator=gen, device="cuda").to(dtype) * 2.0 - 1.0
        return sign * torch.exp2(e)
    return torch.rand(shape, generator=gen, device="cuda", dtype=dtype) * 2.0 - 1.0


def _inputs(case, seed):
    """A, B (and D) of every product, from the seed."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for n, m, p, mode in _problems(case):
        dtype = torch.float64 if MODES[mode][0] == mm.MM_F64 else torch.float32
        a = _values(gen, case["values"], (n, m), dtype)
        b = _values(gen, case["values"], (m, p), dtype)
        d = _values(gen, case["values"], (n, p), dtype) if case["path"] == "axpby" else None
        out.append((a, b, d))
    return out


def _slots(probs):
    """Where a batch's results lie in its output arenas, one arena a type:
    (type, first entry) of each product, 256-byte steps, and the arenas' sizes."""
    ends, slots = {}, []
    for n, _, p, mode in probs:
        dtype = torch.float64 if MODES[mode][0] == mm.MM_F64 else torch.float32
        at = ends.get(dtype, 0)
        slots.append((dtype, at))
        ends[dtype] = at + (n * p + 63) // 64 * 64
    return slots, ends


def _outputs(probs):
    slots, ends = _slots(probs)
    arenas = {t: torch.zeros(e, device="cuda", dtype=t) for t, e in ends.items()}
    outs = [arenas[t][at:at + n * p].view(n, p) for (n, _, p, _), (t, at) in zip(probs, slots)]
    return arenas, outs


def _batch(arenas):
    return [arenas[t] for t in (torch.float32, torch.float64) if t in arenas]


_ready = False


def _library():
    global _ready
    if not _ready:
        mm.check_status(mm.mm_init(device=torch.cuda.current_device()), "mm_init")
        _ready = True


def _stream():
    """The caller's current stream; torch's default stream is CUDA's legacy
    default stream, whose explicit handle is 1."""
    return torch.cuda.current_stream().cuda_stream or 1


def prepare(case, seed):
    _library()
    inputs = _inputs(case, seed)
    probs = _problems(case)
    arenas, outs = _outputs(probs)
    state = {"case": case, "probs": probs, "inputs": inputs, "outs": outs, "arenas": arenas}
    if case["path"] == "grouped":
        state["table"] = mm.mm_problems([(n, m, p, a, b, c) for (n, m, p, _), (a, b, _), c
                                         in zip(probs, inputs, outs)])
    # the serving loop runs on streams of its own: the inputs are complete first
    torch.cuda.synchronize()
    return state


def run(state):
    case, outs = state["case"], state["outs"]
    if case["path"] == "grouped":
        dt, mode = MODES[case["mode"]]
        mm.check_status(mm.mm_gemm_grouped_async(state["table"], dt, mode, _stream()), "grouped")
        return _batch(state["arenas"])
    if case["path"] == "serve":
        ids = []
        for (n, m, p, mode), (a, b, _), c in zip(state["probs"], state["inputs"], outs):
            st, rid = mm.mm_submit(n, m, p, a, b, c, *MODES[mode])
            mm.check_status(st, "submit")
            ids.append(rid)
        for rid in ids:
            st, result, _, _ = mm.mm_wait(rid, 60.0)
            mm.check_status(st, "wait")
            mm.check_status(result, "request")
        return _batch(state["arenas"])
    (n, m, p, mode), (a, b, d), c = state["probs"][0], state["inputs"][0], outs[0]
    dt, md = MODES[mode]
    if case["path"] == "axpby":
        mm.check_status(mm.mm_gemm_axpby_async(n, m, p, case["alpha"], a, b, case["beta"], d, c, dt, md,
                                               _stream()), "axpby")
    else:
        mm.check_status(mm.mm_gemm_async(n, m, p, a, b, c, dt, md, _stream()), "gemm")
    return c


def work(case):
    """Each input read once, each output written once; 2 n m p operations."""
    total_bytes = flops = 0
    for n, m, p, mode in _problems(case):
        size = 8 if MODES[mode][0] == mm.MM_F64 else 4
        total_bytes += size * (n * m + m * p + n * p * (2 if case["path"] == "axpby" else 1))
        flops += 2 * n * m * p
    return {"bytes": total_bytes, "flops": flops}


def exact(case, seed):
    probs, inputs = _problems(case), _inputs(case, seed)
    if case["path"] in ("grouped", "serve"):
        slots, ends = _slots(probs)
        arenas = {t: torch.zeros(e, device="cuda", dtype=torch.float64) for t, e in ends.items()}
        for (n, _, p, _), (a, b, _), (t, at) in zip(probs, inputs, slots):
            arenas[t][at:at + n * p] = (a.double() @ b.double()).reshape(-1)
        return _batch(arenas)
    a, b, d = inputs[0]
    c = a.double() @ b.double()
    if case["path"] == "axpby":
        c = case["alpha"] * c + case["beta"] * d.double()
    return c
