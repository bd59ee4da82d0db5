"""Sparse products C = A * B that users of this library compute, for timing and comparison.

Every case goes through the public entry points: ``Handle.multiply``,
``Handle.symbolic`` / ``Handle.numeric`` over a row window,
``Handle.numeric_values``, the learned sizing mode and ``Batch.run``. Inputs
are drawn on the GPU, with the shapes and value distributions of
``workloads.py``: the structure of a random matrix from the case's own
"graph" number, the values from the seed.
"""

from __future__ import annotations

import json
import math
import random

import numpy as np
import torch

import paper_2206_07244_gb300 as ops
from paper_2206_07244_gb300 import learned
from paper_2206_07244_gb300.batch import Batch

# A call's products, at most: the row slabs in which the benchmark and
# spgemm_multiply_host compute a C that does not fit in memory.
SLAB = 1.5e9


def listed():
    return [
        # The smallest call: one 2D 5-point operator squared, as at the
        # coarse end of a multigrid hierarchy. Latency and launches count.
        {"name": "grid5_64", "kind": "grid5", "nx": 64, "ny": 64},
        # Rectangular factors of unstructured data with unsorted rows, some
        # repeated columns and 64-bit row pointers, sizes that no tile
        # divides.
        {"name": "uniform_unsorted_i64", "kind": "uniform", "m": 60013, "k": 40009, "n": 50021,
         "degree": 12, "sorted": False, "i64": True, "graph": 1},
        # A band matrix (spline or finite-difference operator), middle-sized
        # rows with a high compression ratio.
        {"name": "banded_65", "kind": "banded", "n": 1 << 17, "half_bw": 32},
        # The regular high-compression workload of the benchmark: a 27-point
        # finite-element stencil on 128^3 points.
        {"name": "stencil27_128", "kind": "stencil27", "side": 128, "mode": "plain"},
        # The same operator family in an iterative setup: new coefficients,
        # same structure, only the values of C again. An odd side.
        {"name": "stencil27_95_values", "kind": "stencil27", "side": 95, "mode": "values"},
        # Learned row sizing with the committed predictor.
        {"name": "stencil27_101_learned", "kind": "stencil27", "side": 101, "mode": "learned"},
        # Decoupled subsystems: 1024 dense-ish diagonal blocks, hundreds of
        # entries per row of C.
        {"name": "blocks_1m", "kind": "blocks", "n": 1 << 20, "width": 1024, "degree": 24, "mode": "plain",
         "graph": 7},
        # A power-law graph squared whole (two-hop neighbourhoods).
        {"name": "rmat16", "kind": "rmat", "scale": 16, "degree": 16, "at": 0.0, "products": SLAB, "graph": 1},
        # The benchmark's graph, n = 2^20 and degree 16, one row slab of it.
        {"name": "rmat20_slab", "kind": "rmat", "scale": 20, "degree": 16, "at": 0.5, "products": SLAB, "graph": 1},
        # The benchmark's largest graph, n = 2^21 and degree 32: B is wider
        # than one shared-memory bitmap. One row slab.
        {"name": "rmat21_slab", "kind": "rmat", "scale": 21, "degree": 32, "at": 0.3, "products": SLAB, "graph": 2021},
        # One level of a multigrid setup on a large grid: A P, then P^T (A P).
        {"name": "galerkin_level_128", "kind": "level", "side": 128},
        # 512 uneven Galerkin products in one batch launch.
        {"name": "galerkin_batch_512", "kind": "batch", "count": 512, "lo": 8, "hi": 48, "graph": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid5", "uniform", "uniform", "banded", "stencil27", "stencil27", "blocks", "rmat", "rmat",
                       "rmat", "level", "batch"])
    graph = rng.randint(1, 1 << 20)
    if kind == "grid5":
        return {"kind": kind, "nx": _log_int(rng, 24, 1024), "ny": _log_int(rng, 24, 1024)}
    if kind == "uniform":
        return {"kind": kind, "m": _log_int(rng, 2000, 300000), "k": _log_int(rng, 2000, 300000),
                "n": _log_int(rng, 2000, 300000), "degree": rng.randint(2, 32), "sorted": rng.random() < 0.5,
                "i64": rng.random() < 0.5, "graph": graph}
    if kind == "banded":
        half = rng.randint(1, 65)
        most = min(1 << 20, int(1.2e9 / (2 * half + 1) ** 2))
        return {"kind": kind, "n": _log_int(rng, 4096, most), "half_bw": half}
    if kind == "stencil27":
        return {"kind": kind, "side": _log_int(rng, 12, 128), "mode": rng.choice(["plain", "plain", "values", "learned"])}
    if kind == "blocks":
        return {"kind": kind, "n": _log_int(rng, 1 << 14, 1 << 20), "width": _log_int(rng, 128, 4096),
                "degree": rng.randint(6, 24), "mode": rng.choice(["plain", "plain", "learned"]), "graph": graph}
    if kind == "rmat":
        return {"kind": kind, "scale": rng.randint(12, 21), "degree": rng.randint(4, 32),
                "at": round(rng.random(), 3), "products": float(_log_int(rng, 2e7, SLAB)), "graph": graph}
    if kind == "level":
        return {"kind": kind, "side": _log_int(rng, 12, 150)}
    lo = rng.randint(8, 40)
    return {"kind": kind, "count": _log_int(rng, 16, 512), "lo": lo, "hi": rng.randint(lo, 48), "graph": graph}


# --- inputs ------------------------------------------------------------------

def _gen(seed, part=0):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + part) % (1 << 62))


def _uniform(gen, n, lo, hi):
    return torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _rpt(counts, i64=False):
    rpt = torch.zeros(counts.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(counts, 0, out=rpt[1:])
    return rpt if i64 else rpt.to(torch.int32)


def _stencil(dims, offsets, gen, lo, hi, diagonal):
    """Grid operator: rows are the points of a grid of `dims` (x fastest),
    entries the in-grid neighbours at `offsets` with values uniform in
    [lo, hi] and `diagonal` at the point itself, columns ascending."""
    n = math.prod(dims)
    i = torch.arange(n, device="cuda")
    at, stride, s = [], [], 1
    for d in dims:
        at.append((i // s) % d)
        stride.append(s)
        s *= d
    offsets = sorted(offsets, key=lambda o: sum(a * b for a, b in zip(o, stride)))
    inside = torch.ones((n, len(offsets)), dtype=torch.bool, device="cuda")
    for j, o in enumerate(offsets):
        for p, d, e in zip(at, dims, o):
            if e:
                inside[:, j] &= (p + e >= 0) & (p + e < d)
    shift = torch.tensor([sum(a * b for a, b in zip(o, stride)) for o in offsets], device="cuda")
    col = (i[:, None] + shift)[inside].to(torch.int32)
    rpt = _rpt(inside.sum(1))
    val = _uniform(gen, col.numel(), lo, hi)
    row = torch.repeat_interleave(i.to(torch.int32), (rpt[1:] - rpt[:-1]).long())
    val[col == row] = diagonal
    return ops.CSR(n, n, rpt, col, val)


def _grid5(nx, ny, gen):
    return _stencil((nx, ny), [(0, 0), (-1, 0), (1, 0), (0, -1), (0, 1)], gen, -1.5, -0.5, 4.0)


def _stencil27(side, gen):
    box = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)]
    return _stencil((side,) * 3, box, gen, 0.5, 1.5, 27.0)


def _seven(side, gen):
    faces = [(0, 0, 0)] + [tuple(s if a == b else 0 for b in range(3)) for a in range(3) for s in (-1, 1)]
    return _stencil((side,) * 3, faces, gen, -1.5, -0.5, 6.0)


def _banded(n, half, gen):
    return _stencil((n,), [(o,) for o in range(-half, half + 1)], gen, -1.0, 1.0, 2.0)


def _coo_unique(rows, cols, r, c, values):
    """Entries (r, c) with duplicates merged, values uniform in [-1, 1]."""
    key = torch.unique(r * cols + c)
    r = key // cols
    counts = torch.bincount(r, minlength=rows)
    return ops.CSR(rows, cols, _rpt(counts), (key - r * cols).to(torch.int32), _uniform(values, key.numel(), -1.0, 1.0))


def _rmat(scale, degree, gen, values, a=0.57, b=0.19, c=0.19):
    n, m = 1 << scale, degree << scale
    r = torch.zeros(m, dtype=torch.int64, device="cuda")
    q = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        u = torch.rand(m, generator=gen, device="cuda")
        low = u >= a + b
        right = ((u >= a) & ~low) | (u >= a + b + c)
        r.mul_(2).add_(low)
        q.mul_(2).add_(right)
    return _coo_unique(n, n, r, q, values)


def _blocks(n, width, degree, gen, values):
    """Diagonal blocks of about `width` rows, about `degree` entries a row."""
    count = max(1, n // width)
    bounds = torch.linspace(0, n, count + 1, dtype=torch.float64, device="cuda").long()
    r = torch.arange(n, device="cuda").repeat_interleave(degree)
    blk = torch.bucketize(r, bounds[1:], right=True)
    lo, hi = bounds[blk], bounds[blk + 1]
    u = torch.rand(r.numel(), generator=gen, device="cuda", dtype=torch.float64)
    c = torch.minimum(lo + (u * (hi - lo)).long(), hi - 1)
    return _coo_unique(n, n, r, c, values)


def _random(rows, cols, degree, ordered, i64, gen, values):
    """Row lengths uniform in [0, 2 degree], columns uniform (repeats kept)."""
    counts = torch.randint(0, 2 * degree + 1, (rows,), generator=gen, device="cuda")
    nnz = int(counts.sum())
    col = torch.randint(0, cols, (nnz,), generator=gen, device="cuda")
    if ordered:
        r = torch.repeat_interleave(torch.arange(rows, device="cuda"), counts)
        col = torch.sort(r * cols + col)[0] % cols
    return ops.CSR(rows, cols, _rpt(counts, i64), col.to(torch.int32), _uniform(values, nnz, -1.0, 1.0))


def _prolongator(side):
    """Piecewise-constant prolongation of 2x2x2 aggregates and its transpose."""
    sc = (side + 1) // 2
    i = torch.arange(side ** 3, device="cuda")
    x, y, z = i % side, (i // side) % side, i // (side * side)
    agg = ((z // 2) * sc + y // 2) * sc + x // 2
    P = ops.CSR(side ** 3, sc ** 3, torch.arange(side ** 3 + 1, dtype=torch.int32, device="cuda"),
                agg.to(torch.int32), torch.ones(side ** 3, dtype=torch.float64, device="cuda"))
    order = torch.sort(agg, stable=True)[1]
    PT = ops.CSR(sc ** 3, side ** 3, _rpt(torch.bincount(agg, minlength=sc ** 3)), order.to(torch.int32),
                 torch.ones(side ** 3, dtype=torch.float64, device="cuda"))
    return P, PT


def _nprod(A, B):
    length = (B.rpt[1:] - B.rpt[:-1]).long()
    run = torch.zeros(A.nnz + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(length[A.col.long()], 0, out=run[1:])
    return run[A.rpt.long()]   # products of the rows before each row


def _window(case, A, B):
    """Rows [r0, r1) of about case["products"] products, starting at the
    fraction case["at"] of what does not fit."""
    before = _nprod(A, B)
    total = int(before[-1])
    if total <= case["products"]:
        return 0, A.rows
    first = int(case["at"] * (total - case["products"]))
    edges = torch.tensor([first, first + int(case["products"])], device="cuda")
    r0, r1 = (torch.searchsorted(before, edges, right=True) - 1).tolist()
    return r0, max(r1, r0 + 1)


def _sides(case):
    rng = random.Random(case["graph"])
    return [rng.randint(case["lo"], case["hi"]) for _ in range(case["count"])]


def _inputs(case, seed):
    """A, B and the row window of a single product."""
    kind, values = case["kind"], _gen(seed)
    graph = _gen(case.get("graph", 0), 2)
    if kind == "uniform":
        A = _random(case["m"], case["k"], case["degree"], case["sorted"], case["i64"], graph, values)
        B = _random(case["k"], case["n"], case["degree"], case["sorted"], case["i64"], graph, values)
        return A, B, (0, A.rows)
    if kind == "grid5":
        A = _grid5(case["nx"], case["ny"], values)
    elif kind == "banded":
        A = _banded(case["n"], case["half_bw"], values)
    elif kind == "stencil27":
        A = _stencil27(case["side"], values)
    elif kind == "blocks":
        A = _blocks(case["n"], case["width"], case["degree"], graph, values)
    else:
        A = _rmat(case["scale"], case["degree"], graph, values)
    return A, A, (_window(case, A, A) if kind == "rmat" else (0, A.rows))


def _new_values(A, seed):
    val = A.val * _uniform(_gen(seed, 1), A.nnz, 0.5, 1.5)
    return ops.CSR(A.rows, A.cols, A.rpt, A.col, val)


# --- the cases ---------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind, "handle": ops.Handle()}
    h = state["handle"]
    if kind == "level":
        A = _seven(case["side"], _gen(seed))
        P, PT = _prolongator(case["side"])
        return state | {"A": A, "P": P, "PT": PT}
    if kind == "batch":
        sides = _sides(case)
        As, Ps, PTs = [], [], []
        for i, s in enumerate(sides):
            A = _seven(s, _gen(seed, i))
            P, PT = _prolongator(s)
            As.append(A)
            Ps.append(P)
            PTs.append(PT)
        n = len(sides)
        b = Batch(h, As + PTs, Ps + [None] * n, b_from=[-1] * n + list(range(n)))
        b.run()
        b.sync()
        coarse = [b.result(n + i) for i in range(n)]
        return state | {"batch": b, "coarse": coarse}
    A, B, rows = _inputs(case, seed)
    state |= {"A": A, "B": B, "rows": rows}
    if case.get("mode") == "values":
        state["C"] = h.multiply(A, B)
        state["A"] = state["B"] = _new_values(A, seed)
    elif case.get("mode") == "learned":
        with open(learned.MANIFEST) as f:
            margin = json.load(f)["margin"]
        h.set_predictor(np.load(learned.WEIGHTS), margin)
        h.set_mode("learned")
    return state


def _parts(C):
    return {"rpt": C.rpt, "col": C.col, "val": C.val}


def run(state):
    h = state["handle"]
    if state["kind"] == "level":
        AP = h.multiply(state["A"], state["P"])
        return {"AP": _parts(AP), "coarse": _parts(h.multiply(state["PT"], AP))}
    if state["kind"] == "batch":
        b, coarse = state["batch"], state["coarse"]
        b.run()
        # every coarse operator of the batch, packed behind one another
        out = {"rpt": torch.cat([C.rpt for C in coarse]), "col": torch.cat([C.col for C in coarse]),
               "val": torch.cat([C.val for C in coarse])}
        b.sync()
        return out
    if "C" in state:
        return _parts(h.numeric_values(state["A"], state["B"], state["C"]))
    r0, r1 = state["rows"]
    h.symbolic(state["A"], state["B"], r0, r1)
    return _parts(h.numeric(state["A"], state["B"]))


# --- work --------------------------------------------------------------------


def _product_work(A, B, rows=None):
    """Bytes of A's rows, the referenced rows of B and C, and 2 flops a product."""
    r0, r1 = rows or (0, A.rows)
    before = _nprod(A, B)
    products = int(before[r1] - before[r0])
    e0, e1 = int(A.rpt[r0]), int(A.rpt[r1])
    used = torch.unique(A.col[e0:e1].long())
    b_entries = int((B.rpt[1:] - B.rpt[:-1]).long()[used].sum())
    with ops.Handle() as h:
        nnz = h.symbolic(A, B, r0, r1)
    a_size, b_size = A.rpt.element_size(), B.rpt.element_size()
    read = a_size * (r1 - r0 + 1) + 12 * (e1 - e0) + b_size * used.numel() + 12 * b_entries
    return {"bytes": read + 8 * (r1 - r0 + 1) + 12 * nnz, "flops": 2 * products}


def work(case):
    kind = case["kind"]
    total = {"bytes": 0, "flops": 0}
    if kind in ("level", "batch"):
        sides = [case["side"]] if kind == "level" else _sides(case)
        once = {}
        for s in sorted(set(sides)):
            A = _seven(s, _gen(0))
            P, PT = _prolongator(s)
            with ops.Handle() as h:
                AP = h.multiply(A, P)
            two = _product_work(A, P), _product_work(PT, AP)
            once[s] = {k: two[0][k] + two[1][k] for k in total}
        for s in sides:
            for k in total:
                total[k] += once[s][k]
        return total
    A, B, rows = _inputs(case, 0)
    return _product_work(A, B, rows)


# --- exact values ------------------------------------------------------------

def _exact_product(A, B, rows=None, most=1 << 27):
    """Values of C = A * B in column order: every product expanded, sorted by
    its position in C and summed, `most` products at a time."""
    r0, r1 = rows or (0, A.rows)
    before = _nprod(A, B)
    brpt, arpt = B.rpt.long(), A.rpt.long()
    length = brpt[1:] - brpt[:-1]
    parts, cols, counts = [], [], []
    r = r0
    while r < r1:
        limit = before[r] + most
        e = int(torch.searchsorted(before, limit, right=True)) - 1
        e = min(max(e, r + 1), r1)
        p0, p1 = int(arpt[r]), int(arpt[e])
        k = A.col[p0:p1].long()
        n = length[k]
        run = torch.cumsum(n, 0)
        entry = torch.repeat_interleave(torch.arange(p1 - p0, device="cuda"), n)
        q = torch.arange(entry.numel(), device="cuda") - (run - n)[entry] + brpt[k][entry]
        arow = torch.repeat_interleave(torch.arange(e - r, device="cuda"), arpt[r + 1:e + 1] - arpt[r:e])
        key = arow[entry] * B.cols + B.col[q].long()
        prod = A.val[p0:p1][entry] * B.val[q]
        del q, entry
        key, order = torch.sort(key)
        prod = prod[order]
        del order
        place, where = torch.unique_consecutive(key, return_inverse=True)
        del key
        parts.append(torch.zeros(place.numel(), dtype=torch.float64, device="cuda").index_add_(0, where, prod))
        row = place // B.cols
        cols.append((place - row * B.cols).to(torch.int32))
        counts.append(torch.bincount(row, minlength=e - r))
        r = e
    if not parts:
        return ops.CSR(0, B.cols, _rpt(torch.zeros(0, dtype=torch.int64, device="cuda"), True), B.col[:0], B.val[:0])
    return ops.CSR(r1 - r0, B.cols, _rpt(torch.cat(counts), True), torch.cat(cols), torch.cat(parts))


def exact(case, seed):
    kind = case["kind"]
    if kind == "level":
        A = _seven(case["side"], _gen(seed))
        P, PT = _prolongator(case["side"])
        AP = _exact_product(A, P)
        coarse = _exact_product(PT, AP)
        return {"AP": {"rpt": None, "col": None, "val": AP.val}, "coarse": {"rpt": None, "col": None, "val": coarse.val}}
    if kind == "batch":
        vals = []
        for i, s in enumerate(_sides(case)):
            P, PT = _prolongator(s)
            vals.append(_exact_product(PT, _exact_product(_seven(s, _gen(seed, i)), P)).val)
        return {"rpt": None, "col": None, "val": torch.cat(vals)}
    A, B, rows = _inputs(case, seed)
    if case.get("mode") == "values":
        A = B = _new_values(A, seed)
    return {"rpt": None, "col": None, "val": _exact_product(A, B, rows).val}
