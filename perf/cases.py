"""Performance cases of the reduction-to-all: what they are, their inputs, one
pass through the public entry points, the work a pass cannot do without and
its result in 64 bits.

A case names an entry point (``path``), the rank count ``p``, the vector
length ``m``, the element kind, the topology, the block count ``b`` (0: the
plan's default, -1: blocks of 16000 elements, as in the paper's experiment)
and whether the rank rows are ``packed`` one behind the other (a dense [p, m]
array, whose rows start on 16-byte boundaries only when m allows) or each
start on a 256-byte boundary, as separately allocated buffers do.
"""
from __future__ import annotations

import math

import torch

import paper_2109_12626_gb300 as pkg

ESIZE = {"int32": 4, "float32": 4, "mat2x2u32": 16, "mat2x2f32": 16}
# operations per element and combine: one sum, or 2x2 by 2x2 (8 products, 4 sums)
OPS = {"int32": 1, "float32": 1, "mat2x2u32": 12, "mat2x2f32": 12}
PAPER_BLOCK = 16000  # elements per pipeline block in the paper's Table 2 runs


def _case(name, path, p, m, kind, b=0, topology="dual", packed=False):
    return {"name": name, "path": path, "p": p, "m": m, "kind": kind, "b": b,
            "topology": topology, "packed": packed}


def listed():
    return [
        # a handful of ranks with short vectors (a few scalars or a bias per
        # worker): launch and call latency
        _case("fused_p7_m1000_int32", "fused", 7, 1000, "int32"),
        # many ranks with short vectors (histograms, counters): latency of a
        # deep tree
        _case("fused_p1152_m1024_int32", "fused", 1152, 1024, "int32"),
        # one of the paper's counts, in a dense [p, m] array whose rows start
        # 8 bytes off a 16-byte boundary: ragged and unaligned
        _case("fused_p288_m21250_int32_packed", "fused", 288, 21250, "int32", packed=True),
        # the non-commutative operator on a mid-size problem
        _case("fused_p36_m65536_mat2x2u32", "fused", 36, 65536, "mat2x2u32"),
        # the middle of the paper's range of counts at its full rank count
        _case("fused_p1152_m65536_int32", "fused", 1152, 65536, "int32"),
        # gradients of a few million parameters over many ranks
        _case("fused_p1152_m4194304_f32", "fused", 1152, 4194304, "float32"),
        # gradients of a large model over a few ranks (the benchmark's default)
        _case("fused_p32_m134217728_f32", "fused", 32, 134217728, "float32"),
        # Algorithm 1 on short vectors at the paper's rank count
        _case("schedule_p288_m250_int32", "schedule", 288, 250, "int32"),
        # Algorithm 1 in the middle range, default block count
        _case("schedule_p1152_m65536_int32", "schedule", 1152, 65536, "int32"),
        # Algorithm 1 on long vectors, a set block count
        _case("schedule_p32_m8388608_f32", "schedule", 32, 8388608, "float32", b=16),
        # the pipelined reduce, then broadcast, in the paper's comparison:
        # 16000-element blocks
        _case("reduce_bcast_p288_m875000_int32", "reduce_bcast", 288, 875000, "int32", b=-1,
              topology="single"),
        # host buffers in, host buffers out
        _case("host_p36_m65536_mat2x2f32", "host", 36, 65536, "mat2x2f32"),
    ]


def draw(rng):
    path = rng.choice(["fused"] * 7 + ["schedule"] * 3 + ["reduce_bcast", "host"])
    kind = rng.choice(["int32", "float32", "int32", "float32", "mat2x2u32", "mat2x2f32"])
    p = int(round(math.exp(rng.uniform(math.log(2), math.log(1152)))))
    most = 1 << (32 if path == "fused" else 29 if path == "host" else 30)  # bytes of inputs
    total = math.exp(rng.uniform(math.log(4096), math.log(most)))
    m = max(1, int(total / (p * ESIZE[kind])))
    b = 0
    if path in ("schedule", "reduce_bcast"):
        b = rng.choice([0, 0, -1, int(round(math.exp(rng.uniform(0, math.log(512)))))])
        b = min(b, m)
    topology = "single" if path == "reduce_bcast" or rng.random() < 0.15 else "dual"
    c = _case("", path, p, m, kind, b, topology, rng.random() < 0.25)
    del c["name"]
    return c


def _blocks(case):
    return -(-case["m"] // PAPER_BLOCK) if case["b"] < 0 else case["b"]


def _rows(case, device, pin=False):
    """[p, m] (matrices: [p, m, 4]) of uninitialised rank rows."""
    words = case["m"] * ESIZE[case["kind"]] // 4
    pitch = words if case["packed"] else -(-words // 64) * 64
    dt = torch.float32 if case["kind"] in ("float32", "mat2x2f32") else torch.int32
    base = torch.empty((case["p"], pitch), dtype=dt, device=device, pin_memory=pin)[:, :words]
    return base.unflatten(1, (case["m"], 4)) if case["kind"].startswith("mat") else base


def _fill(case, x, seed):
    """The seeded inputs, made on the device x lives on."""
    g = torch.Generator(device=x.device)
    g.manual_seed(seed)
    kind = case["kind"]
    if kind == "int32":      # counters: [-2^20, 2^20], sums may wrap
        x.random_(-(1 << 20), (1 << 20) + 1, generator=g)
    elif kind == "float32":  # gradient-like
        x.normal_(0.0, 1e-3, generator=g)
    elif kind == "mat2x2u32":  # full words, products mod 2^32
        x.random_(-(1 << 31), 1 << 31, generator=g)
    else:                    # near the identity, so long products stay in range
        x.uniform_(-(2.0**-7), 2.0**-7, generator=g)
        x[..., 0] += 1.0
        x[..., 3] += 1.0


def prepare(case, seed):
    host = case["path"] == "host"
    x = _rows(case, "cuda")
    _fill(case, x, seed)
    if host:
        xh = _rows(case, "cpu", pin=True)
        xh.copy_(x)
        x = xh
        y = _rows(case, "cpu", pin=True)
    else:
        y = _rows(case, "cuda")
    y.zero_()
    plan = pkg.Plan(case["p"], case["m"], case["kind"], _blocks(case), case["topology"])
    xs, ys = list(x.unbind(0)), list(y.unbind(0))
    call = None
    if not host:
        bound = plan.bind(xs, ys)
        call = {"fused": bound.allreduce, "schedule": bound.allreduce_schedule,
                "reduce_bcast": bound.allreduce_reduce_bcast}[case["path"]]
    return {"plan": plan, "x": x, "y": y, "xs": xs, "ys": ys, "call": call}


def run(state):
    if state["call"] is not None:
        state["call"]()
    else:
        state["plan"].allreduce_host(state["xs"], state["ys"])
    return state["y"]


def work(case):
    n = case["p"] * case["m"]
    return {"bytes": 2 * n * ESIZE[case["kind"]],
            "flops": (case["p"] - 1) * case["m"] * OPS[case["kind"]]}


def tolerance(case):
    # every entry point keeps the bracketing of the trees, so each result has
    # one right bit pattern, whatever the kernel and the block count
    return "exact"


def exact(case, seed):
    x = _rows(case, "cuda")
    _fill(case, x, seed)
    kind, p = case["kind"], case["p"]
    wide = torch.float64 if kind in ("float32", "mat2x2f32") else torch.int64
    acc = x[0].to(wide)
    for i in range(1, p):
        v = x[i].to(wide)
        if kind in ("int32", "float32"):
            acc += v
            continue
        a, b, c, d = acc.unbind(-1)
        e, f, g, h = v.unbind(-1)
        acc = torch.stack((a * e + b * g, a * f + b * h, c * e + d * g, c * f + d * h), -1)
        if wide is torch.int64:  # keep the low 32 bits, signed
            acc = ((acc + (1 << 31)) & 0xFFFFFFFF) - (1 << 31)
    if wide is torch.int64:
        acc = (((acc + (1 << 31)) & 0xFFFFFFFF) - (1 << 31)).to(torch.int32)
    out = acc.unsqueeze(0).expand((p,) + tuple(acc.shape))
    return out.cpu() if case["path"] == "host" else out
