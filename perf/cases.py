"""The cases this framework's speed is judged on: one call each of its public
entry points, over the sizes, element types and options that programs use.

Kinds and what they stand for in a program:

* ``region``       one `reduction(...)` loop over an array (accr_reduce)
* ``rows``         a gang/vector nest with one variable per row (accr_rowreduce)
* ``matmul``       the Listing-1a matrix nest, in the mode the caller picks
* ``batch``        many independent regions in one call (accr_batch_reduce)
* ``segments``     consecutive segments of one array (accr_segmented_reduce)
* ``nearest``      k nearest points of a query (accr_nearest_k)
* ``standardize``  SRAD's statistics and the elementwise region they feed
* ``bfs``          level-synchronous search with a convergence flag

A case's shape (lengths of regions and segments included) follows from the
case alone; the values come from the seed.
"""
import math

import numpy as np
import torch

from paper_1412_1127_gb300 import _native, api

DEV = "cuda"
DTYPE = {"i32": torch.int32, "i64": torch.int64, "f32": torch.float32, "f64": torch.float64}
SIZE = {"i32": 4, "i64": 8, "f32": 4, "f64": 8}


def listed():
    return [
        # the smallest call: a 4 MiB loop with a sum and a maximum, where the launch and the merge count
        {"name": "region_small", "kind": "region", "elem": "i32", "n": 1 << 20, "off": 0,
         "clauses": "add:i64 max:i32", "comp": False},
        # a float array summed into a double variable, of no round length and starting mid-vector
        {"name": "region_wide", "kind": "region", "elem": "f32", "n": 10000019, "off": 1,
         "clauses": "add:f64 max:f32", "comp": False},
        # one pass over a 1 GiB array for its compensated sum and its range
        {"name": "region_large", "kind": "region", "elem": "f32", "n": 1 << 28, "off": 0,
         "clauses": "add:f32 max:f32 min:f32", "comp": True},
        # many short rows of an odd length (a table of records): sum and maximum of each
        {"name": "rows_narrow", "kind": "rows", "elem": "f32", "rows": 400000, "cols": 61, "pad": 0,
         "clauses": "add:f32 max:f32", "comp": False},
        # a few medium rows of a padded double matrix: sum and minimum of each
        {"name": "rows_few", "kind": "rows", "elem": "f64", "rows": 100, "cols": 30001, "pad": 7,
         "clauses": "add:f64 min:f64", "comp": False},
        # the paper's own matrix product, 1024 x 1024, in float on the CUDA cores
        {"name": "matmul_simt", "kind": "matmul", "mode": "simt", "len": 1024},
        # the large matrix nest on the tensor cores, operands split in the call
        {"name": "matmul_bf16x3", "kind": "matmul", "mode": "bf16x3", "len": 4096},
        # 20,000 independent loops of very different lengths in one call
        {"name": "batch", "kind": "batch", "regions": 20000, "hi": 1 << 17},
        # the short segments of a sparse matrix's rows: sum and maximum of each
        {"name": "segments", "kind": "segments", "elem": "f32", "nseg": 100000, "hi": 1 << 10,
         "clauses": "add:f32 max:f32", "comp": False},
        # the ten records nearest to a position, ten million records
        {"name": "nearest", "kind": "nearest", "n": 10000001, "k": 10},
        # SRAD's image step: mean and variance of a 16 MiB image, then the standardised image
        {"name": "standardize", "kind": "standardize", "n": 1 << 22},
        # breadth-first search of a maze of 1024 x 1024 cells until nothing changes
        {"name": "bfs", "kind": "bfs", "mode": "persistent", "rows": 1024, "cols": 1024, "open": 0.62},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


REGION_CLAUSES = [("i32", "add:i64 max:i32", False), ("i32", "add:i32", False), ("i32", "max:i32 min:i32", False),
                  ("i32", "bxor:i32", False), ("i64", "add:i64 bxor:i64", False), ("f32", "add:f32", False),
                  ("f32", "add:f32", True), ("f32", "add:f32 max:f32", True), ("f32", "add:f32 max:f32 min:f32", True),
                  ("f32", "add:f64", False), ("f32", "add:f64 max:f32", False), ("f64", "add:f64", False),
                  ("f64", "add:f64 max:f64 min:f64", False)]
ROW_CLAUSES = [("f32", "add:f32 max:f32", False), ("f32", "add:f32", True), ("f32", "add:f64", False),
               ("f64", "add:f64 min:f64", False), ("i32", "add:i64 max:i32", False), ("i64", "add:i64", False)]
SEGMENT_CLAUSES = [("f32", "add:f32 max:f32", False), ("f32", "add:f32", True), ("f64", "add:f64", False),
                   ("i32", "add:i64", False), ("i64", "add:i64 bxor:i64", False)]


def draw(rng):
    kind = rng.choice(["region", "region", "rows", "rows", "matmul", "batch", "segments", "nearest", "standardize", "bfs"])
    if kind == "region":
        elem, clauses, comp = rng.choice(REGION_CLAUSES)
        return {"kind": kind, "elem": elem, "n": _log_int(rng, 1 << 14, (1 << 30) // SIZE[elem]), "off": rng.randrange(4),
                "clauses": clauses, "comp": comp}
    if kind == "rows":
        elem, clauses, comp = rng.choice(ROW_CLAUSES)
        total = _log_int(rng, 1 << 18, (1 << 28) // SIZE[elem])
        cols = _log_int(rng, 4, min(total, 1 << 20))
        return {"kind": kind, "elem": elem, "rows": max(1, total // cols), "cols": cols, "pad": rng.choice([0, 0, 3, 8]),
                "clauses": clauses, "comp": comp}
    if kind == "matmul":
        mode = rng.choice(["simt", "serial", "bf16x3", "bf16x3"])
        return {"kind": kind, "mode": mode, "len": _log_int(rng, 200, 4096 if mode == "bf16x3" else 2048)}
    if kind == "batch":
        return {"kind": kind, "regions": _log_int(rng, 500, 20000), "hi": _log_int(rng, 1 << 8, 1 << 17)}
    if kind == "segments":
        elem, clauses, comp = rng.choice(SEGMENT_CLAUSES)
        nseg = _log_int(rng, 1000, 200000)
        hi = _log_int(rng, 16, min(1 << 16, max(32, (1 << 28) // nseg)))
        return {"kind": kind, "elem": elem, "nseg": nseg, "hi": hi, "clauses": clauses, "comp": comp}
    if kind == "nearest":
        return {"kind": kind, "n": _log_int(rng, 1 << 15, 1 << 26), "k": rng.randint(1, 16)}
    if kind == "standardize":
        return {"kind": kind, "n": _log_int(rng, 1 << 16, 1 << 27)}
    if rng.random() < 0.3:  # the form the host drives, level by level
        return {"kind": kind, "mode": "reduce", "rows": rng.randint(48, 200), "cols": rng.randint(48, 200),
                "open": round(rng.uniform(0.65, 0.95), 3)}
    return {"kind": kind, "mode": "persistent", "rows": _log_int(rng, 64, 1024), "cols": _log_int(rng, 64, 1024),
            "open": round(rng.uniform(0.62, 0.95), 3)}


# ---- inputs -----------------------------------------------------------------------


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _values(elem, n, g):
    if elem == "f32":
        return torch.randn(n, generator=g, device=DEV, dtype=torch.float32)
    if elem == "f64":
        return torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
    if elem == "i32":
        return torch.randint(-(1 << 31), 1 << 31, (n,), generator=g, device=DEV, dtype=torch.int32)
    return torch.randint(-(1 << 40), 1 << 40, (n,), generator=g, device=DEV, dtype=torch.int64)


def _pairs(text):
    return [tuple(c.split(":")) for c in text.split()]


def _outs(clauses, n):
    return [torch.zeros(n, dtype=DTYPE[acc], device=DEV) for _, acc in _pairs(clauses)]


def _lengths(count, lo, hi):
    """Lengths log-uniform on [lo, hi], in an order fixed by the case."""
    r = np.random.Generator(np.random.PCG64([count, hi]))
    v = np.exp(r.uniform(math.log(lo), math.log(hi), size=count))
    return np.clip(np.ceil(v).astype(np.int64), lo, hi)


def _offsets(lengths):
    return np.concatenate([np.zeros(1, dtype=np.int64), np.cumsum(lengths)])


def _prepare_region(c, g):
    x = _values(c["elem"], c["n"] + c["off"], g)[c["off"]:]
    outs = _outs(c["clauses"], 1)
    return {"x": x, "outs": outs, "clauses": [api.clause(op, o) for (op, _), o in zip(_pairs(c["clauses"]), outs)],
            "flags": api.ACCR_COMPENSATED if c["comp"] else 0}


def _prepare_rows(c, g):
    ld = c["cols"] + c["pad"]
    A = _values(c["elem"], c["rows"] * ld, g).view(c["rows"], ld)[:, :c["cols"]]
    outs = _outs(c["clauses"], c["rows"])
    return {"A": A, "outs": outs, "clauses": [api.clause(op, o) for (op, _), o in zip(_pairs(c["clauses"]), outs)],
            "flags": api.ACCR_COMPENSATED if c["comp"] else 0}


def _prepare_matmul(c, g):
    n = c["len"]
    a, b = (torch.rand(n, n, generator=g, device=DEV) * 2 - 1 for _ in range(2))
    return {"a": a, "b": b, "c": torch.empty_like(a), "mode": c["mode"]}


def _prepare_batch(c, g):
    """Even regions: float N(0,1), compensated +; odd ones: int64, + and ^."""
    lengths = _lengths(c["regions"], 1, c["hi"])
    off_f, off_i = _offsets(lengths[0::2]), _offsets(lengths[1::2])
    nf, ni = len(off_f) - 1, len(off_i) - 1
    f, i = _values("f32", int(off_f[-1]), g), _values("i64", int(off_i[-1]), g)
    sf = torch.zeros(nf, device=DEV)
    si, xi = (torch.zeros(ni, dtype=torch.int64, device=DEV) for _ in range(2))
    regions = []
    for k in range(c["regions"]):
        j = k // 2
        if k % 2 == 0:
            regions.append((f[off_f[j]:off_f[j + 1]], [api.clause("add", sf[j:j + 1])], api.ACCR_COMPENSATED))
        else:
            regions.append((i[off_i[j]:off_i[j + 1]], [api.clause("add", si[j:j + 1]), api.clause("bxor", xi[j:j + 1])], 0))
    desc, keep = api.regions_array(regions)  # a C program's own array of descriptors
    return {"f": f, "i": i, "off_f": off_f, "desc": desc, "keep": keep, "count": c["regions"], "outs": [sf, si, xi]}


def _prepare_segments(c, g):
    off = _offsets(_lengths(c["nseg"], 1, c["hi"]))
    outs = _outs(c["clauses"], c["nseg"])
    return {"x": _values(c["elem"], int(off[-1]), g), "off": off, "outs": outs,
            "clauses": [api.clause(op, o) for (op, _), o in zip(_pairs(c["clauses"]), outs)],
            "flags": api.ACCR_COMPENSATED if c["comp"] else 0}


def _prepare_nearest(c, g):
    q = np.random.default_rng(int(g.initial_seed())).uniform(10, 90, size=2)
    return {"pts": torch.rand(c["n"], 2, generator=g, device=DEV) * 100, "q": (float(q[0]), float(q[1])), "k": c["k"],
            "idx": torch.empty(c["k"], dtype=torch.int64, device=DEV), "d2": torch.empty(c["k"], device=DEV)}


def _prepare_standardize(c, g):
    x = torch.randn(c["n"], generator=g, device=DEV) * 3 + 5
    return {"x": x, "y": torch.empty_like(x), "stats": torch.empty(2, dtype=torch.float64, device=DEV)}


def _prepare_bfs(c, g):
    """Random cells, with a short open street around the source so that it
    seldom starts in a closed pocket."""
    rows, cols = c["rows"], c["cols"]
    cells = (torch.rand(rows, cols, generator=g, device=DEV) < c["open"]).to(torch.uint8)
    r, q = rows // 2, cols // 2
    cells[r, max(0, q - 24):q + 25] = 1
    return {"open": cells, "src": r * cols + q, "mode": c["mode"],
            "dist": torch.empty(rows, cols, dtype=torch.int32, device=DEV)}


def prepare(case, seed):
    return dict({"region": _prepare_region, "rows": _prepare_rows, "matmul": _prepare_matmul, "batch": _prepare_batch,
                 "segments": _prepare_segments, "nearest": _prepare_nearest, "standardize": _prepare_standardize,
                 "bfs": _prepare_bfs}[case["kind"]](case, _gen(seed)), kind=case["kind"])


# ---- one pass -----------------------------------------------------------------------


def run(s):
    kind = s["kind"]
    if kind == "region":
        api.accr_reduce(s["x"], s["clauses"], flags=s["flags"])
        return s["outs"]
    if kind == "rows":
        api.accr_rowreduce(s["A"], s["clauses"], flags=s["flags"])
        return s["outs"]
    if kind == "matmul":
        api.accr_matmul_nest(s["a"], s["b"], s["c"], mode=s["mode"])
        return s["c"]
    if kind == "batch":
        _native.check(_native.lib().accr_batch_reduce(s["desc"], s["count"], 0, torch.cuda.current_stream().cuda_stream))
        return s["outs"]
    if kind == "segments":
        api.accr_segmented_reduce(s["x"], s["off"], s["clauses"], flags=s["flags"])
        return s["outs"]
    if kind == "nearest":
        api.accr_nearest_k(s["pts"], s["q"][0], s["q"][1], s["k"], s["idx"], s["d2"])
        return {"idx": s["idx"], "d2": s["d2"]}
    if kind == "standardize":
        api.accr_standardize(s["x"], s["y"], s["stats"])
        return {"y": s["y"], "stats": s["stats"]}
    levels = api.accr_grid_bfs(s["open"], s["src"], s["dist"], mode=s["mode"])
    return {"dist": s["dist"], "levels": levels}


# ---- what a pass cannot do without ---------------------------------------------------


def work(c):
    """Bytes: each input read once, each output written once.  Flops: one per
    element and clause (the nest: a multiply and an add per term; the nearest
    points: the distance)."""
    kind = c["kind"]
    if kind == "region":
        return {"bytes": c["n"] * SIZE[c["elem"]], "flops": c["n"] * len(_pairs(c["clauses"]))}
    if kind == "rows":
        n = c["rows"] * c["cols"]
        out = sum(SIZE[a] for _, a in _pairs(c["clauses"]))
        return {"bytes": n * SIZE[c["elem"]] + c["rows"] * out, "flops": n * len(_pairs(c["clauses"]))}
    if kind == "matmul":
        # BF16x3 multiplies three pairs of bf16 operands for each float product
        return {"bytes": 12 * c["len"] ** 2, "flops": (6 if c["mode"] == "bf16x3" else 2) * c["len"] ** 3}
    if kind == "batch":
        L = _lengths(c["regions"], 1, c["hi"])
        nf, ni = int(L[0::2].sum()), int(L[1::2].sum())
        return {"bytes": 4 * nf + 8 * ni + 4 * len(L[0::2]) + 16 * len(L[1::2]), "flops": nf + 2 * ni}
    if kind == "segments":
        n = int(_lengths(c["nseg"], 1, c["hi"]).sum())
        out = sum(SIZE[a] for _, a in _pairs(c["clauses"]))
        return {"bytes": n * SIZE[c["elem"]] + c["nseg"] * (8 + out), "flops": n * len(_pairs(c["clauses"]))}
    if kind == "nearest":
        return {"bytes": 8 * c["n"], "flops": 5 * c["n"]}
    if kind == "standardize":
        return {"bytes": 8 * c["n"], "flops": 5 * c["n"]}
    return {"bytes": 5 * c["rows"] * c["cols"], "flops": 0}


# ---- the same in 64 bits ---------------------------------------------------------------


def _exact_fold(op, x, dim=None):
    """One clause over a float tensor; None for whole-number results."""
    if not x.is_floating_point():
        return None
    if op == "add":
        return x.double().sum().reshape(1) if dim is None else x.double().sum(dim)
    f = torch.amax if op == "max" else torch.amin
    return f(x).double().reshape(1) if dim is None else f(x, dim).double()


def _exact_segments(op, x, off):
    if not x.is_floating_point():
        return None
    lengths = torch.from_numpy(np.diff(off)).to(DEV)
    ids = torch.repeat_interleave(torch.arange(len(off) - 1, device=DEV), lengths)
    if op == "add":
        return torch.zeros(len(off) - 1, dtype=torch.float64, device=DEV).index_add_(0, ids, x.double())
    r = torch.full((len(off) - 1,), -math.inf if op == "max" else math.inf, dtype=torch.float64, device=DEV)
    return r.scatter_reduce_(0, ids, x.double(), "amax" if op == "max" else "amin")


def exact(case, seed):
    kind = case["kind"]
    if case.get("elem", "f32") in ("i32", "i64") or kind == "bfs":
        return None  # whole numbers only
    s = prepare(case, seed)
    if kind == "region":
        return [_exact_fold(op, s["x"]) for op, _ in _pairs(case["clauses"])]
    if kind == "rows":
        return [_exact_fold(op, s["A"], 1) for op, _ in _pairs(case["clauses"])]
    if kind == "matmul":
        return s["a"].double() @ s["b"].double()
    if kind == "batch":
        return [_exact_segments("add", s["f"], s["off_f"]), None, None]
    if kind == "segments":
        return [_exact_segments(op, s["x"], s["off"]) for op, _ in _pairs(case["clauses"])]
    if kind == "nearest":
        d = s["pts"].double() - torch.tensor(np.float32(s["q"]), device=DEV).double()
        return {"idx": None, "d2": torch.topk(d.square().sum(1), s["k"], largest=False).values}
    x = s["x"].double()
    mean = x.mean()
    var = (x * x).mean() - mean * mean
    return {"y": (x - mean) / var.sqrt(), "stats": torch.stack([mean, var])}
