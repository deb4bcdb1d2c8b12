"""What a program that uses this framework has it do, as cases that can be timed.

The work is the triplet merge tree of a float32 field on a regular grid and
what is read off it: trees with their persistence pairs and the components of
a sublevel set (one call, or call by call), re-queries of a finished tree with
short branches removed, branch decompositions, batches of uneven fields,
trees with 64-bit vertex ids, and requests sent to the server. Field kinds
and sizes are those of the benchmark, the tests and the generators of
``paper_2301_10838_gb300.fields``: white noise, Gaussian random fields
quantised to 12 bits (many ties), lognormal density-like fields.

Pair lists and branch offsets are as long as the field's minima: their
buffers are zeroed before the call and come back whole.

Every output is whole numbers (vertex ids), so there is no 64-bit reference
value to be near to: outputs are equal or wrong.
"""

from __future__ import annotations

import math
import random

import torch

import paper_2301_10838_gb300 as mt
from paper_2301_10838_gb300 import fields
from paper_2301_10838_gb300.batch import Batch
from paper_2301_10838_gb300.serve import Server

# local minima per vertex of each field kind, for the size of the pair list
_MINIMA = {"white": 1.0 / 7.0, "lognormal": 0.1, "grf_q12": 0.05, "grf": 0.05}


def listed():
    return [
        # one small noisy block at a time, as in a loop over time steps or
        # tiles of an image: launches and latency count
        {"name": "step_white_64", "kind": "step", "field": "white", "nx": 64, "ny": 64, "nz": 64, "q": 0.3},
        # an ordinary simulation volume stored with 12 bits: ties everywhere
        {"name": "step_grf_q12_256", "kind": "step", "field": "grf_q12", "nx": 256, "ny": 256, "nz": 256, "q": 0.5},
        # a cropped scan: sides that are no multiple of anything, odd rows
        {"name": "step_ragged_509", "kind": "step", "field": "lognormal", "nx": 509, "ny": 430, "nz": 333, "q": 0.5},
        # the headline volume: density-like, 1.07e9 vertices
        {"name": "step_lognormal_1024", "kind": "step", "field": "lognormal", "nx": 1024, "ny": 1024, "nz": 1024,
         "q": 0.5},
        # call by call on the superlevel sets (the split tree): the tree, its
        # pairs, then the components above a threshold
        {"name": "calls_split_512", "kind": "calls", "field": "lognormal", "nx": 512, "ny": 512, "nz": 512, "q": 0.8},
        # a finished tree queried again: pairs and components with the
        # branches below a persistence removed
        {"name": "requery_simplified_400", "kind": "requery", "field": "lognormal", "nx": 400, "ny": 400, "nz": 400,
         "q": 0.6, "eps": 0.05},
        # every vertex grouped by branch: a small volume and an ordinary one
        {"name": "branches_grf_q12_128", "kind": "branches", "field": "grf_q12", "nx": 128, "ny": 128, "nz": 128},
        {"name": "branches_lognormal_512", "kind": "branches", "field": "lognormal", "nx": 512, "ny": 512, "nz": 512},
        # 512 fields of uneven sizes in one graph replay
        {"name": "batch_uneven_512", "kind": "batch", "count": 512, "lo": 16, "hi": 128, "sizes": 7},
        # the calls for grids past 2^32 vertices, on a volume that leaves
        # room for other work on the card
        {"name": "wide_lognormal_512", "kind": "wide", "field": "lognormal", "nx": 512, "ny": 512, "nz": 512, "q": 0.5},
        # a burst of requests of mixed sizes from host memory to the server
        {"name": "serve_burst_16", "kind": "serve", "count": 16, "lo": 32, "hi": 256, "sizes": 11},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "calls", "requery", "branches", "batch", "wide", "serve"])
    if kind == "batch":
        return {"kind": kind, "count": _log_int(rng, 16, 512), "lo": 16, "hi": rng.randint(32, 128),
                "sizes": rng.randrange(1 << 20)}
    if kind == "serve":
        return {"kind": kind, "count": rng.randint(4, 16), "lo": 32, "hi": rng.randint(64, 256),
                "sizes": rng.randrange(1 << 20)}
    top = {"step": 768, "calls": 640, "requery": 640, "branches": 512, "wide": 512}[kind]
    side = _log_int(rng, 32, top)
    case = {"kind": kind, "field": rng.choice(["white", "lognormal", "grf_q12"])}
    for axis in ("nx", "ny", "nz"):
        # sides within a factor of the drawn one, odd ones among them; some
        # are rounded to multiples of 16 as simulation grids are
        s = min(1024, max(8, int(round(side * math.exp(rng.uniform(-0.3, 0.3))))))
        case[axis] = max(16, s // 16 * 16) if rng.random() < 0.4 else s
    if kind != "branches":
        case["q"] = round(rng.uniform(0.1, 0.9), 3)
    if kind == "requery":
        case["eps"] = round(rng.uniform(0.0, 0.2), 3)
    return case


def _field(kind, shape, seed):
    """A float32 field on the GPU: (nz, ny, nx)."""
    if kind == "white":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        return torch.rand(shape, generator=gen, dtype=torch.float32, device="cuda")
    if kind == "lognormal":
        return fields.lognormal(shape, seed, 0.8, -2.0, device="cuda")
    if kind == "grf":
        return fields.grf(shape, -2.5, seed, device="cuda")
    g = fields.grf(shape, -3.0, seed, device="cuda")
    lo, hi = g.min(), g.max()
    return torch.round((g - lo) * (4095.0 / (hi - lo).clamp_min(1e-30))) / 4095.0


def _threshold(f, q):
    """About the q-quantile of f, from a sample of its values."""
    flat = f.reshape(-1)
    step = max(1, flat.numel() // 1_000_003)
    return float(torch.quantile(flat[::step][:1_000_000].float(), q))


def _sizes(case):
    """Cube sides of the server's requests, log-uniform in [lo, hi]."""
    rng = random.Random(case["sizes"])
    return [_log_int(rng, case["lo"], case["hi"]) for _ in range(case["count"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        shapes = fields.batch_shapes(case["count"], case["lo"], case["hi"], case["sizes"])
        b = Batch(shapes)
        for i, s in enumerate(shapes):
            if i < len(shapes) // 2:
                b.field(i).copy_(_field("white", s, 1000 * seed + i))
            else:
                b.field(i).copy_(fields.grf(s, -3.0, 1000 * seed + i, device="cuda"))
        b.pairs.zero_()  # fields write only as many pairs as they have
        b.capture()
        return {"kind": kind, "batch": b}
    if kind == "serve":
        reqs = []
        for i, side in enumerate(_sizes(case)):
            f = _field("grf", (side, side, side), 1000 * seed + i)
            n = f.numel()
            reqs.append((f.cpu().pin_memory(), _threshold(f, 0.2 + 0.6 * ((7 * i) % 10) / 10.0),
                         torch.zeros((n // 2 + 1, 2), dtype=torch.int32, pin_memory=True),
                         torch.empty(n, dtype=torch.int32, pin_memory=True)))
        return {"kind": kind, "server": Server(hbm_budget_bytes=2 << 30, max_slots=8), "requests": reqs}
    f = _field(case["field"], (case["nz"], case["ny"], case["nx"]), seed)
    n, grid = f.numel(), mt.grid_of(f)
    st = {"kind": kind, "f": f, "t": _threshold(f, case["q"]) if "q" in case else 0.0}
    if kind == "wide":
        st["grid"] = grid
        st["ws"] = mt.wide_workspace(grid)
        st["W"] = torch.empty((n, 2), dtype=torch.int64, device="cuda")
        st["pairs"] = torch.zeros((n // 2 + 1, 2), dtype=torch.int64, device="cuda")
        st["labels"] = torch.empty(n, dtype=torch.int64, device="cuda")
        return st
    st["W"] = torch.empty(n, dtype=torch.int64, device="cuda")
    if kind in ("requery", "branches"):  # the tree is in hand
        build_ws = mt.workspace(grid)
        mt.mt_build_triplets(f, st["W"], build_ws)
        mt.mt_sync_status(build_ws)
    if kind == "branches":
        st["ws"] = mt.branches_workspace(grid)
        st["order"] = torch.empty(n, dtype=torch.int32, device="cuda")
        st["offsets"] = torch.zeros(n // 2 + 2, dtype=torch.int32, device="cuda")
        return st
    st["ws"] = mt.workspace(grid)
    st["pairs"] = torch.zeros((n // 2 + 1, 2), dtype=torch.int32, device="cuda")
    st["labels"] = torch.empty(n, dtype=torch.int32, device="cuda")
    st["eps"] = case.get("eps", 0.0)
    return st


def run(st):
    kind = st["kind"]
    if kind == "step":
        k, root = mt.mt_build_step(st["f"], st["W"], st["t"], st["labels"], st["pairs"], st["ws"])
        return {"W": st["W"], "labels": st["labels"], "pairs": st["pairs"], "npairs": k, "root": root}
    if kind == "calls":
        mt.mt_build_triplets_ex(st["f"], st["W"], st["ws"], mt.MT_SUPERLEVEL)
        k, root = mt.mt_persistence_pairs(st["f"], st["W"], st["pairs"], st["ws"])
        mt.mt_components_at_ex(st["f"], st["W"], st["t"], mt.MT_SUPERLEVEL, st["labels"], st["ws"])
        return {"W": st["W"], "labels": st["labels"], "pairs": st["pairs"], "npairs": k, "root": root}
    if kind == "requery":
        k, root = mt.mt_simplified_pairs(st["f"], st["W"], st["eps"], 0, st["pairs"], st["ws"])
        mt.mt_simplified_components_at(st["f"], st["W"], st["t"], st["eps"], 0, st["labels"], st["ws"])
        return {"labels": st["labels"], "pairs": st["pairs"], "npairs": k, "root": root}
    if kind == "branches":
        k = mt.mt_branch_decomposition(st["f"], st["W"], 0, st["order"], st["offsets"], st["ws"])
        return {"order": st["order"], "offsets": st["offsets"], "branches": k}
    if kind == "wide":
        mt.mt_build_triplets_wide(st["f"], st["W"], st["ws"])
        k, root = mt.mt_persistence_pairs_wide(st["W"], st["grid"], st["pairs"], st["ws"])
        mt.mt_components_at_wide(st["f"], st["W"], st["t"], 0, st["labels"], st["ws"])
        return {"W": st["W"], "labels": st["labels"], "pairs": st["pairs"], "npairs": k, "root": root}
    if kind == "batch":
        b = st["batch"]
        b.launch()
        return {"W": b.W, "pairs": b.pairs, "npairs": b.npairs}
    srv = st["server"]
    tickets = [srv.submit(f, t, pairs=pairs, labels=labels) for f, t, pairs, labels in st["requests"]]
    done = [srv.wait(k) for k in tickets]
    return {"labels": [d["labels"] for d in done], "pairs": [r[2] for r in st["requests"]],
            "npairs": torch.tensor([d["npairs"] for d in done]), "roots": torch.tensor([d["root"] for d in done])}


def work(case):
    """Bytes of one pass: each input read once, each output written once."""
    kind = case["kind"]
    if kind == "batch":
        ns = [a * b * c for a, b, c in fields.batch_shapes(case["count"], case["lo"], case["hi"], case["sizes"])]
        n = sum(ns)
        return {"bytes": 12 * n + 8 * 0.1 * n, "flops": 0}
    if kind == "serve":
        n = sum(s ** 3 for s in _sizes(case))
        # host to device and back: the field in, the labels and pairs out
        return {"bytes": 8 * n + 8 * _MINIMA["grf"] * n, "flops": 0}
    n = case["nx"] * case["ny"] * case["nz"]
    m = _MINIMA[case["field"]] * n
    per_vertex, per_pair = {
        "step": (4 + 8 + 4, 8),       # field in; triplets, labels, pairs out
        "calls": (4 + 8 + 4, 8),
        "requery": (4 + 8 + 4, 8),    # field and triplets in; labels, pairs out
        "branches": (4 + 8 + 4, 4),   # field and triplets in; order, offsets out
        "wide": (4 + 16 + 8, 16),
    }[kind]
    return {"bytes": per_vertex * n + per_pair * m, "flops": 0}
