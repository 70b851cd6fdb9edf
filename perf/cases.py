"""What the time of this framework is measured on: calls of the public binding (`zccl.Context`) as programs that move
scientific fields and gradients make them, from a 4 KiB message to a 1 GiB array.

The inputs have the distributions of `paper_2502_18554_b200/fields.py` (sums of sinusoids with noise, a random field of
64 cosine modes, Laplace-distributed gradients with exact zeros and outliers), made on the GPU from the seed alone.  A
program keeps ONE context and calls it for many arrays, and so does this file: states of equally sized cases share it.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2502_18554_b200 import zccl as z

# Bits per value of the compressed streams, for work(): (distribution, bound) -> approximate size.
BITS = {("smooth", 1e-2): 1.6, ("smooth", 1e-3): 2.3, ("smooth", 1e-4): 4.2,
        ("field", 1e-2): 2.8, ("field", 1e-3): 5.3, ("field", 1e-4): 8.5,
        ("gradient", 1e-5): 9.8}


def listed():
    return [
        # a 4 KiB message of a latency-bound exchange, relative bound (the default way to state a bound)
        {"name": "compress 1Ki rel", "op": "compress", "n": 1 << 10, "data": "smooth", "mode": "rel", "eb": 1e-3},
        # the receiving side of a small message
        {"name": "decompress 16Ki", "op": "decompress", "n": 1 << 14, "data": "smooth", "eb": 1e-3},
        # one step of a ring on a short, ragged chunk: decompress, add the local chunk, compress again
        {"name": "hop 100003", "op": "hop", "n": 100_003, "data": "smooth", "eb": 1e-3, "reduce": "sum", "raw": False},
        # a 256^3 field, one array after another: what a simulation writes out per variable and step
        {"name": "compress 16Mi field rel", "op": "compress", "n": 1 << 24, "data": "field", "mode": "rel", "eb": 1e-3},
        # reading such a field back, at the tightest of the usual bounds
        {"name": "decompress 16Mi field", "op": "decompress", "n": 1 << 24, "data": "field", "eb": 1e-4},
        # a ring step on a large chunk
        {"name": "hop 16Mi field", "op": "hop", "n": 1 << 24, "data": "field", "eb": 1e-3, "reduce": "sum", "raw": False},
        # a 1 GiB gradient bucket at a tight absolute bound (code lengths of 7 to 15 bits)
        {"name": "compress 256Mi gradient", "op": "compress", "n": 1 << 28, "data": "gradient", "mode": "abs", "eb": 1e-5},
        # a large array whose length is no multiple of anything
        {"name": "decompress 67110221", "op": "decompress", "n": (1 << 26) + 1357, "data": "smooth", "eb": 1e-3},
        # ring Allreduce over 8 ranks, 8 MiB each (whole collective, emulated in one GPU's memory)
        {"name": "allreduce 8x2Mi", "op": "allreduce", "n": 1 << 21, "ranks": 8, "data": "smooth", "eb": 1e-3},
        # ring Allgather over 8 ranks, 1 MiB each
        {"name": "allgather 8x256Ki", "op": "allgather", "n": 1 << 18, "ranks": 8, "data": "smooth", "eb": 1e-3},
        # double-precision simulation output, there and back
        {"name": "f64 pair 8Mi", "op": "f64", "n": (1 << 23) + 5, "data": "field", "mode": "rel", "eb": 1e-4},
        # arrays in pinned host memory, compressed and restored through the host-buffer calls
        {"name": "host pair 16Mi", "op": "host", "n": 1 << 24, "data": "field", "mode": "rel", "eb": 1e-3},
    ]


def _length(rng, lo, hi):
    """Log-uniform over [lo, hi]; two out of three are odd lengths, the others a multiple of 32."""
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    return max(32, n & ~31) if rng.random() < 1 / 3 else n | 1


def draw(rng: random.Random):
    op = rng.choice(["compress", "compress", "decompress", "decompress", "hop", "hop", "allreduce", "allgather", "f64", "host"])
    lo, hi = {"compress": (1 << 10, 1 << 27), "decompress": (1 << 10, 1 << 27), "hop": (1 << 10, 1 << 25), "allreduce": (1 << 13, 1 << 22),
              "allgather": (1 << 10, 1 << 21), "f64": (1 << 13, 1 << 24), "host": (1 << 13, 1 << 24)}[op]
    n = _length(rng, lo, hi)
    data = rng.choice(["smooth", "field", "gradient"] if n >= 1 << 18 else ["smooth", "gradient"])
    case = {"op": op, "n": n, "data": data}
    if op in ("compress", "f64", "host"):
        case["mode"] = "abs" if data == "gradient" else rng.choice(["rel", "rel", "abs"])
    case["eb"] = 1e-5 if data == "gradient" else rng.choice([1e-2, 1e-3, 1e-4])
    if op == "hop":
        case["reduce"] = rng.choice(["sum", "sum", "sum", "max"])
        case["raw"] = rng.random() < 0.25
    if op in ("allreduce", "allgather"):
        case["ranks"] = rng.randint(2, 8)
    return case


# ---------------------------------------------------------------------------------------------- inputs

def _array(kind: str, n: int, seed: int, dtype=torch.float32) -> torch.Tensor:
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = random.Random(seed)
    if kind == "gradient":   # Laplace(0, 1e-3), 10 % exact zeros, 0.1 % outliers from N(0, 0.1)
        u = torch.rand(n, device="cuda", generator=g)
        v = u.sub_(0.5).sign() * torch.log1p(u.abs_().mul_(-2.0).clamp_(min=-0.9999999)).mul_(-1e-3)
        u = torch.rand(n, device="cuda", generator=g)
        v = torch.where(u < 0.1, torch.zeros((), device="cuda"), v)
        out = torch.where(u > 0.999, torch.randn(n, device="cuda", generator=g).mul_(0.1), v)
        return out.to(dtype)
    if kind == "smooth":     # three sinusoids and noise of 1e-3
        i = torch.arange(n, device="cuda", dtype=torch.float64)
        v = torch.randn(n, device="cuda", generator=g, dtype=torch.float64).mul_(1e-3)
        for _ in range(3):
            a, p, ph = r.uniform(0.5, 2.0), r.uniform(1e3, 1e5), r.uniform(0.0, 2 * math.pi)
            v += (i * (2 * math.pi / p) + ph).sin_().mul_(a)
        return v.to(dtype)
    # 64 cosine modes of a cube, integer wave vectors 1 <= |k| <= 16, amplitude |k|^-2, noise of 1e-4; row-major.  A mode
    # is a product of functions of (x, y) and of z, so the field is one small matrix product.
    side = max(2, math.ceil(round(n ** (1 / 3), 6)))
    rows = -(-n // side)
    ks = []
    while len(ks) < 64:
        k = [r.randint(-16, 16) for _ in range(3)]
        kn = math.sqrt(sum(c * c for c in k))
        if 1.0 <= kn <= 16.0:
            ks.append((*k, kn ** -2.0, r.uniform(0.0, 2 * math.pi)))
    t = torch.tensor(ks, device="cuda", dtype=torch.float64)
    w = 2 * math.pi / side
    row = torch.arange(rows, device="cuda")
    xy = (torch.outer((row // side).double(), t[:, 0]) + torch.outer((row % side).double(), t[:, 1])) * w + t[:, 4]
    zz = torch.outer(t[:, 2], torch.arange(side, device="cuda", dtype=torch.float64)) * w
    v = (xy.cos() * t[:, 3]) @ zz.cos() - (xy.sin() * t[:, 3]) @ zz.sin()
    v = v.reshape(-1)[:n]
    v = v + torch.randn(n, device="cuda", generator=g, dtype=torch.float64).mul_(1e-4)
    return v.to(dtype).contiguous()


_kept: dict = {}


def _context(elems: int, ranks: int = 0) -> z.Context:
    """The program's context: one, kept as long as the sizes stay the same."""
    if (elems, ranks) not in _kept:
        _kept.clear()
        _kept[elems, ranks] = z.Context(elems, ranks)
    return _kept[elems, ranks]


def _absolute(x: torch.Tensor, case: dict) -> float:
    """The case's bound as an absolute one (what the ranks of a collective have agreed on before)."""
    return case["eb"] if case["data"] == "gradient" else case["eb"] * float((x.max() - x.min()).item())


def _stream_buffers(n: int):
    return (torch.zeros(z.compress_bound(n), dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda"))


def prepare(case: dict, seed: int):
    op, n, data = case["op"], case["n"], case["data"]
    s = {"op": op}
    if op in ("allreduce", "allgather"):
        ranks = case["ranks"]
        s["ctx"] = _context(n if op == "allreduce" else n * ranks, ranks)
        s["send"] = [_array(data, n, seed * 1009 + k) for k in range(ranks)]
        s["recv"] = [torch.zeros(n if op == "allreduce" else n * ranks, device="cuda") for _ in range(ranks)]
        s["mode"], s["eb"] = (z.EB_ABS if data == "gradient" else z.EB_REL), case["eb"]
        return s
    s["ctx"] = _context(n)
    x = _array(data, n, seed * 1009, torch.float64 if op == "f64" else torch.float32)
    if op in ("compress", "f64", "host"):
        s["mode"] = z.EB_REL if case["mode"] == "rel" else z.EB_ABS
        s["eb"] = case["eb"] if case["mode"] == "rel" else _absolute(x, case)
    if op == "compress":
        s["x"] = x
        s["out"], s["bytes"] = _stream_buffers(n)
    elif op == "f64":
        s["x"], s["y"] = x, torch.zeros_like(x)
        s["out"], s["bytes"] = _stream_buffers(n)
    elif op == "host":
        s["x"] = x.cpu().pin_memory()
        s["out"] = torch.zeros(z.compress_bound(n), dtype=torch.uint8).pin_memory()
        s["y"] = torch.zeros(n).pin_memory()
    else:   # decompress, hop: an incoming stream
        s["in"], got = _stream_buffers(n)
        eb = _absolute(x, case)
        s["ctx"].compress(x, z.EB_ABS, eb, s["in"], got)
        s["in"] = s["in"][: int(got.item())].clone()
        if op == "decompress":
            s["y"] = torch.zeros(n, device="cuda")
        else:
            s["n"], s["local"] = n, _array(data, n, seed * 1009 + 1)
            s["out"], s["bytes"] = _stream_buffers(n)
            s["raw"] = torch.zeros(n, device="cuda") if case["raw"] else None
            s["flags"] = z.OP_MAX if case["reduce"] == "max" else z.OP_SUM
    return s


# ---------------------------------------------------------------------------------------------- one pass

def run(s):
    op, ctx = s["op"], s["ctx"]
    if op == "compress":
        ctx.compress(s["x"], s["mode"], s["eb"], s["out"], s["bytes"])
        return s["out"], s["bytes"]
    if op == "decompress":
        ctx.decompress(s["in"], s["y"])
        return s["y"]
    if op == "hop":
        ctx.decompress_reduce_compress(s["in"], s["n"], s["out"], s["bytes"], local=s["local"], raw_out=s["raw"], flags=s["flags"])
        return s["out"], s["bytes"], s["raw"]
    if op == "allreduce":
        ctx.sim_allreduce(s["send"], s["recv"], s["mode"], s["eb"])
        return s["recv"]
    if op == "allgather":
        ctx.sim_allgather(s["send"], s["recv"], s["mode"], s["eb"])
        return s["recv"]
    if op == "f64":
        ctx.compress_f64(s["x"], s["mode"], s["eb"], s["out"], s["bytes"])
        ctx.decompress_f64(s["out"], s["y"])
        return s["out"], s["bytes"], s["y"]
    size = ctx.compress_host(s["x"], s["mode"], s["eb"], s["out"])
    ctx.decompress_host(s["out"], size, s["y"])
    return s["out"], size, s["y"]


# ---------------------------------------------------------------------------------------------- what a pass is about

def work(case: dict) -> dict:
    """Each input read once, each output written once; per value and codec direction a multiplication, a rounding, a
    difference or sum and the code (counted as 4 operations)."""
    op, n = case["op"], case["n"]
    packed = n * BITS[case["data"], case["eb"]] / 8
    if op in ("compress", "decompress"):
        return {"bytes": 4 * n + packed, "flops": 4 * n}
    if op == "hop":
        return {"bytes": 4 * n + 2 * packed + (4 * n if case["raw"] else 0), "flops": 9 * n}
    if op == "allreduce":     # every rank's array in, every rank's result out; each chunk passes the codec once per rank and way
        return {"bytes": 8 * n * case["ranks"], "flops": (9 + 4) * n * case["ranks"]}
    if op == "allgather":
        return {"bytes": 4 * n * case["ranks"] * (1 + case["ranks"]), "flops": 4 * n * case["ranks"] * case["ranks"]}
    if op == "f64":
        return {"bytes": 2 * (8 * n + packed), "flops": 8 * n}
    return {"bytes": 2 * (4 * n + packed), "flops": 8 * n}


def tolerance(case: dict):
    """Streams and reconstructions are defined bit for bit (IEEE operations, no contraction)."""
    return "exact"
