"""Workloads of the library, as its users run them, for timing and for comparing results.

A case is a dict of plain values.  `prepare` makes what a program holds before the call (points, batches,
queries, an index), `run` makes one pass through the public entry points of ``paper_2601_05347_gb300.psi`` and
returns the results, `work` states the bytes and operations the pass cannot do without.

Workloads follow the package's generators (``gen.py``: Uniform, Varden random walks; 2D coordinates of 30 bits, 3D of
21), drawn on the GPU so that inputs of 1e8 points are made in milliseconds.
"""
from __future__ import annotations

import math

import torch

from paper_2601_05347_gb300 import psi

DEV = "cuda"
BITS = {2: 30, 3: 21}
STEP = {2: 1 << 10, 3: 1 << 4}  # Varden step per coordinate
CLUSTERS, RESTART = 100, 1e-4


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the headline build: 1e8 clustered 2D points in walk order into a Hilbert SPaC tree
        dict(name="build_spac_h_2d_1e8", op="build", kind="spac_h", dim=2, data="varden", n=100_000_000, leaf=32),
        # an orth-tree over randomly ordered 3D points (its points come back leaf by leaf, as an exporter reads them)
        dict(name="build_porth_3d_1e7", op="build", kind="porth", dim=3, data="uniform", n=10_000_019, leaf=32),
        # a small whole session, where launches and host calls count: build, insert, delete, k-NN, range count
        dict(name="session_2d_2e4", op="session", kind="spac_h", dim=2, data="varden", n=20_000, leaf=32, m=2_000,
             q=500, k=10, boxes=200, target=100),
        # a tick of a live index: a small batch arrives, is asked around, and expires
        dict(name="tick_spac_h_2d_1e4", op="tick", kind="spac_h", dim=2, data="varden", n=10_000_019, leaf=32,
             batch="near", m=10_000, q=1_000, k=10),
        # the index built by consecutive batches of a tenth (the paper's incremental construction)
        dict(name="incremental_spac_z_3d_5e6", op="incremental", kind="spac_z", dim=3, data="uniform", n=5_000_000,
             leaf=32, slices=10, q=100_000, k=10),
        # the same tick on an orth-tree, a batch of one per cent
        dict(name="tick_porth_3d_5e4", op="tick", kind="porth", dim=3, data="uniform", n=5_000_011, leaf=32,
             batch="near", m=50_000, q=1_000, k=10),
        # the headline query: 1e7 10-NN at data points of a 1e8-point index
        dict(name="knn10_spac_h_2d_1e7", op="knn", kind="spac_h", dim=2, data="varden", n=100_000_000, leaf=32,
             q=10_000_000, k=10, at="data"),
        # long neighbour lists in 3D
        dict(name="knn100_spac_z_3d_2e5", op="knn", kind="spac_z", dim=3, data="varden", n=10_000_000, leaf=32,
             q=200_003, k=100, at="data"),
        # a served query batch of ordinary size: a thousand 10-NN queries, where latency counts
        dict(name="knn10_porth_3d_1e3", op="knn", kind="porth", dim=3, data="uniform", n=1_000_003, leaf=32, q=1_000,
             k=10, at="uniform"),
        # 5e4 boxes of about a thousand points: their counts, and their ids in ascending order
        dict(name="range_spac_h_2d_5e4", op="range", kind="spac_h", dim=2, data="varden", n=20_000_000, leaf=32,
             boxes=50_000, target=1_000),
        # float coordinates (no curve keys): build, 10-NN and range counts
        dict(name="float_3d_3e6", op="float", dim=3, data="uniform", n=3_000_017, leaf=32, q=300_000, k=10,
             boxes=20_000, target=1_000),
        # many small independent indexes in one persistent launch, then 10-NN on all of them
        dict(name="batch_2d_256", op="batch", kind="spac_h", dim=2, data="varden", indexes=256, lo=1_000,
             hi=1_000_000, leaf=32, share=0.1, k=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("build", "build", "session", "tick", "tick", "incremental", "knn", "knn", "knn", "range",
                     "float", "batch"))
    c = dict(op=op, dim=rng.choice((2, 3)), data=rng.choice(("uniform", "varden")),
             leaf=rng.choice((32, 32, 32, 16, 40, 64)))
    if op != "float":
        c["kind"] = rng.choice(("spac_h", "spac_z") if op == "batch" else ("spac_h", "spac_z", "porth"))
    k = rng.choice((1, 5, 10, 10, 10, 32, 100))
    if op == "build":
        c.update(n=_log(rng, 1e4, 3e7))
    elif op == "session":
        n = _log(rng, 2e3, 2e5)
        c.update(n=n, m=max(1, n // rng.choice((10, 50))), q=_log(rng, 10, 4e3), k=k, boxes=_log(rng, 10, 1e3),
                 target=100)
    elif op == "tick":
        n = _log(rng, 2e5, 1e7)
        c.update(n=n, batch=rng.choice(("near", "walk")), m=_log(rng, 100, n / 50), q=_log(rng, 50, 2e3), k=k)
    elif op == "incremental":
        n = _log(rng, 1e5, 5e6)
        c.update(n=n, slices=rng.choice((5, 10, 20)), q=_log(rng, 1e3, 1e5), k=min(k, 10))
    elif op == "knn":
        c.update(n=_log(rng, 1e5, 2e7), q=_log(rng, 300, 1e6 if k <= 32 else 1e5), k=k,
                 at=rng.choice(("data", "uniform")))
    elif op == "range":
        c.update(n=_log(rng, 1e5, 2e7), boxes=_log(rng, 1e3, 5e4), target=rng.choice((10, 100, 1000)))
    elif op == "float":
        c.update(dim=rng.choice((2, 3, 4, 5)), n=_log(rng, 5e4, 3e6), q=_log(rng, 1e3, 2e5), k=min(k, 32),
                 boxes=_log(rng, 100, 2e4), target=100)
    else:
        c.update(indexes=_log(rng, 16, 256), lo=1_000, hi=_log(rng, 1e4, 3e5), share=0.1, k=min(k, 32))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed & 0x7FFFFFFFFFFF)
    return g


def _uniform(n, dim, g):
    return torch.randint(0, 1 << BITS[dim], (n, dim), dtype=torch.int32, device=DEV, generator=g)


def _varden(n, dim, g):
    """Folded random walks (gen.py's recipe): each walker makes a contiguous share of the points and restarts at a
    uniform position with a small probability."""
    full = 1 << BITS[dim]
    start = torch.rand(n, device=DEV, generator=g) < RESTART
    start[(torch.arange(CLUSTERS, device=DEV) * n + CLUSTERS - 1) // CLUSTERS] = True
    start[0] = True
    seg = torch.cumsum(start, 0) - 1
    first = torch.nonzero(start).flatten()
    out = torch.empty((n, dim), dtype=torch.int32, device=DEV)
    for d in range(dim):
        at = torch.randint(0, full, (first.numel(),), device=DEV, generator=g)
        s = torch.randint(-STEP[dim], STEP[dim] + 1, (n,), device=DEV, generator=g)
        s[first] = 0
        cs = torch.cumsum(s, 0)
        t = torch.remainder(cs + (at - cs[first])[seg], 2 * (full - 1))
        out[:, d] = torch.where(t > full - 1, 2 * (full - 1) - t, t).to(torch.int32)
    return out


def _points(data, n, dim, g):
    return _varden(n, dim, g) if data == "varden" and n >= CLUSTERS else _uniform(n, dim, g)


def _ids(n, first=0):
    return torch.arange(first, first + n, dtype=torch.int32, device=DEV)


def _pick(pts, m, g):
    return pts[torch.randint(0, pts.shape[0], (m,), device=DEV, generator=g)]


def _near(pts, m, dim, g):
    """Points a step away from data points: where moving objects go next."""
    p = _pick(pts, m, g)
    return torch.clamp(p + torch.randint(-STEP[dim], STEP[dim] + 1, p.shape, dtype=torch.int32, device=DEV, generator=g),
                       0, (1 << BITS[dim]) - 1)


def _half_side(pts, target, g):
    """Half side of cubes at data points that hold about `target` points (median over 64 centres, on a sample)."""
    n = pts.shape[0]
    take = min(n, 2_000_000)
    sub = pts if take == n else _pick(pts, take, g)
    rank = max(1, min(take, round(target * take / n)))
    centre = _pick(pts, 64, g)
    far = torch.stack([(sub.to(torch.float64) - c).abs().amax(1).kthvalue(rank).values for c in centre.to(torch.float64)])
    return far.median()


def _boxes(pts, q, target, dim, g):
    h = int(_half_side(pts, target, g))
    c = _pick(pts, q, g).to(torch.int64)
    top = (1 << BITS[dim]) - 1
    return torch.cat([(c - h).clamp(0, top), (c + h).clamp(0, top)], 1).to(torch.int32).contiguous()


def _index(c, pts, ids):
    return psi.Index(pts, ids, kind=c["kind"], leaf_size=c["leaf"])


def prepare(case, seed):
    g, c, op = _gen(seed), case, case["op"]
    if op == "batch":
        # sizes spread evenly over their logarithm, large and small ones mixed
        N = c["indexes"]
        sizes = [int(c["lo"] * (c["hi"] / c["lo"]) ** ((i * 7919 % N) / max(1, N - 1))) for i in range(N)]
        off = [0]
        for s in sizes:
            off.append(off[-1] + int(s))
        qn = [max(1, int(s * c["share"])) for s in sizes]
        qoff = [0]
        for s in qn:
            qoff.append(qoff[-1] + s)
        pts = torch.cat([_points(c["data"], int(s), c["dim"], g) for s in sizes])
        q = torch.cat([_pick(pts[off[i]:off[i + 1]], qn[i], g) for i in range(len(sizes))])
        ids = torch.cat([_ids(int(s)) for s in sizes])
        b = psi.Batch(off, dim=c["dim"], kind=c["kind"], leaf_size=c["leaf"])
        b.reserve(qoff[-1])
        return dict(op=op, b=b, pts=pts, ids=ids, q=q, qoff=torch.tensor(qoff, device=DEV), k=c["k"])
    n, dim = c["n"], c["dim"]
    if op == "float":
        pts = (torch.rand((n, dim), device=DEV, generator=g) if c["data"] == "uniform" or dim > 3 else
               (_points("varden", n, dim, g).to(torch.float64) / (1 << BITS[dim])).to(torch.float32).clamp(0, 0.99999994))
        q = _pick(pts, c["q"], g)
        h, ctr = _half_side(pts, c["target"], g).to(torch.float32), _pick(pts, c["boxes"], g)
        return dict(op=op, pts=pts, ids=_ids(n), q=q, boxes=torch.cat([ctr - h, ctr + h], 1).contiguous(), k=c["k"],
                    leaf=c["leaf"], dim=dim)
    pts, ids = _points(c["data"], n, dim, g), _ids(n)
    s = dict(op=op, case=c, pts=pts, ids=ids)
    if op in ("session", "tick"):
        m = c["m"]
        s["new"] = _points(c["data"], m, dim, g) if c.get("batch") == "walk" else _near(pts, m, dim, g)
        s["new_ids"] = _ids(m, n)
        s["deleted"] = torch.zeros(1, dtype=torch.int64, device=DEV)
    if op == "session":
        gone = torch.randperm(n, device=DEV, generator=g)[:c["m"]]
        s.update(gone=pts[gone].contiguous(), gone_ids=ids[gone].contiguous(), q=_pick(pts, c["q"], g),
                 boxes=_boxes(pts, c["boxes"], c["target"], dim, g))
    elif op == "tick":
        s.update(ix=_index(c, pts, ids), q=_pick(s["new"], c["q"], g))
    elif op == "incremental":
        s["q"] = _pick(pts[: n // 2], c["q"], g)
    elif op == "knn":
        s.update(ix=_index(c, pts, ids), q=_pick(pts, c["q"], g) if c["at"] == "data" else _uniform(c["q"], dim, g))
    elif op == "range":
        s.update(ix=_index(c, pts, ids), boxes=_boxes(pts, c["boxes"], c["target"], dim, g),
                 out=torch.zeros(6 * c["boxes"] * c["target"], dtype=torch.int32, device=DEV))
    if op in ("tick", "knn", "range"):  # the index holds its own copy of the points
        del s["pts"], s["ids"]
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    op = s["op"]
    if op == "knn":
        return s["ix"].knn(s["q"], s["case"]["k"])
    if op == "tick":
        ix = s["ix"]
        ix.insert(s["new"], s["new_ids"])
        near = ix.knn(s["q"], s["case"]["k"])
        ix.delete(s["new"], s["new_ids"], s["deleted"])
        return {"near": near, "deleted": s["deleted"], "size": len(ix)}
    if op == "range":
        # the order of a box's ids is only defined with sort=True
        off, ids = s["ix"].range_report(s["boxes"], sort=True)
        total = min(ids.numel(), s["out"].numel())
        s["out"][:total] = ids[:total]  # the program's own result buffer, of one size for every call
        return {"counts": s["ix"].range_count(s["boxes"]), "offsets": off, "ids": s["out"]}
    if op == "batch":
        s["b"].build(s["pts"], s["ids"])
        return s["b"].knn(s["q"], s["qoff"], s["k"])
    if op == "float":
        ix = psi.FOrth(s["pts"], s["ids"], [0.0] * s["dim"], [1.0] * s["dim"], leaf_size=s["leaf"])
        ids, d2 = ix.knn(s["q"], s["k"])
        return {"nodes": ix.num_nodes, "ids": ids, "d2": d2, "counts": ix.range_count(s["boxes"])}
    c = s["case"]
    if op == "build":
        ix = _index(c, s["pts"], s["ids"])
        return (ix.points(), ix.num_nodes) if c["kind"] == "porth" else ix.leaves()
    if op == "session":
        ix = _index(c, s["pts"], s["ids"])
        ix.insert(s["new"], s["new_ids"])
        ix.delete(s["gone"], s["gone_ids"], s["deleted"])
        return {"knn": ix.knn(s["q"], c["k"]), "counts": ix.range_count(s["boxes"]), "deleted": s["deleted"],
                "points": ix.points()}
    n, cut = c["n"], [c["n"] * i // c["slices"] for i in range(c["slices"] + 1)]
    ix = _index(c, s["pts"][: cut[1]], s["ids"][: cut[1]])
    half = None
    for i in range(1, c["slices"]):
        ix.insert(s["pts"][cut[i]: cut[i + 1]], s["ids"][cut[i]: cut[i + 1]])
        if i + 1 == (c["slices"] + 1) // 2:
            half = ix.knn(s["q"], c["k"])
    return {"half": half, "points": ix.points()}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _knn_work(q, k, dim, n):
    """Queries read, k (id, distance) pairs written, every point that some list holds read once (at most all)."""
    return q * (4 * dim + 12 * k) + min(n, q * k) * (4 * dim + 4), q * k * 3 * dim


def work(case):
    c, op, dim = case, case["op"], case["dim"]
    if op == "batch":
        mean = (c["hi"] - c["lo"]) / math.log(c["hi"] / c["lo"])
        n = int(c["indexes"] * mean)
        b, f = _knn_work(int(n * c["share"]), c["k"], dim, n)
        return {"bytes": 2 * n * (4 * dim + 4) + b, "flops": f}
    n, pt = c["n"], 4 * dim + 4  # a point and its id
    if op == "build":
        return {"bytes": 2 * n * pt, "flops": 0}
    if op == "knn":
        b, f = _knn_work(c["q"], c["k"], dim, n)
        return {"bytes": b, "flops": f}
    if op == "range":  # ids written once, the points inside read once (at most all), counts and offsets
        got = c["boxes"] * c["target"]
        return {"bytes": c["boxes"] * (8 * dim + 16) + 4 * got + min(n, got) * pt, "flops": 2 * dim * got}
    if op == "tick":  # the batch read twice and stored once
        b, f = _knn_work(c["q"], c["k"], dim, n)
        return {"bytes": 3 * c["m"] * pt + b, "flops": f}
    b, f = _knn_work(c["q"], c["k"], dim, n)
    if op == "float":
        return {"bytes": 2 * n * pt + b + c["boxes"] * (8 * dim + 8), "flops": f}
    if op == "session":
        return {"bytes": 2 * n * pt + 4 * c["m"] * pt + b + c["boxes"] * (8 * dim + 8), "flops": f}
    return {"bytes": 2 * n * pt + b, "flops": f}


def exact(case, seed):
    """Float distances by brute force in 64 bits, where that is quick; every other result is whole numbers."""
    if case["op"] != "float" or case["q"] * case["n"] > 4e10:
        return None
    s = prepare(case, seed)
    k, pts = case["k"], s["pts"].double()
    d2 = torch.empty((case["q"], k), dtype=torch.float64, device=DEV)
    rows = max(1, int(2e8) // case["n"])
    for a in range(0, case["q"], rows):
        q = s["q"][a: a + rows].double()
        d = torch.zeros((q.shape[0], case["n"]), dtype=torch.float64, device=DEV)
        for j in range(case["dim"]):
            d += (q[:, j, None] - pts[None, :, j]) ** 2
        d2[a: a + rows] = d.topk(k, dim=1, largest=False, sorted=True).values
    return {"nodes": None, "ids": None, "d2": d2, "counts": None}
