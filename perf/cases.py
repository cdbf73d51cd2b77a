"""Timed cases of the library: what a program that uses it calls, over the range of sizes it calls it with.

Every case runs through the public entry points of ``paper_2201_02789_gb300.nestpar`` with the
configuration a program passes (the library default, or the form ``bench.py`` times for that
workload). Inputs are drawn on the GPU from the seed alone, with the shapes of
``paper_2201_02789_gb300/gen.py``: R-MAT digraphs with the Graph500 probabilities, Zipf(2.1)
digraphs, road grids with weights in [1, 255], and Bezier control points uniform in [0, 1)^2 as
multiples of 2^-24.
"""
import math

import numpy as np
import torch

from paper_2201_02789_gb300 import nestpar as npb

DEV = "cuda:0"
NEVER = npb.INT32_MAX   # a threshold above every child count
_CONTEXT = None


def _context():
    """The program's context: one per process, kept (workspace and graph cache live in it)."""
    global _CONTEXT
    if _CONTEXT is None:
        _CONTEXT = npb.Context(0)
    return _CONTEXT


class _Kept:
    """A batch or server handle, destroyed with the state that holds it."""

    def __init__(self, handle, destroy):
        self.handle, self._destroy = handle, destroy

    def __del__(self):
        self._destroy(self.handle)


# ------------------------------------------------------------------------------ cases

def listed():
    return [
        # a small skewed web-like graph: launch latency and short levels decide
        {"name": "bfs-zipf-4096", "kind": "bfs", "graph": "zipf", "n": 4096, "degree": 4},
        # an ordinary small graph of ragged size
        {"name": "sssp-rmat-13007", "kind": "sssp", "graph": "rmat", "n": 13007, "degree": 12},
        # the full-size social-network traversals (16.8 M edges), library default form
        {"name": "bfs-rmat-2e20", "kind": "bfs", "graph": "rmat", "n": 1 << 20, "degree": 16},
        {"name": "sssp-rmat-2e20", "kind": "sssp", "graph": "rmat", "n": 1 << 20, "degree": 16},
        # a road network: hundreds of levels with little work in each
        {"name": "sssp-road-514", "kind": "sssp", "graph": "road", "n": 514 * 514, "degree": 6},
        # shortest paths from several sources of one graph in one call
        {"name": "sssp-multi-16", "kind": "sssp-multi", "graph": "rmat", "n": 1 << 18, "degree": 16, "queries": 16},
        # many unequal instances solved in one launch
        {"name": "batch-bfs-40", "kind": "batch-bfs", "count": 40, "log2_lo": 10.0, "log2_hi": 17.0},
        # a burst of queries served over two resident graphs
        {"name": "serve-48", "kind": "serve", "n": 1 << 16, "degree": 16, "queries": 48},
        # tessellation: a handful of shapes, a drawing, a large drawing (25 M points, more than L2
        # holds); the default form and the form without a child grid
        {"name": "bezier-1000", "kind": "bezier", "curves": 1000, "threshold": 32, "parent_block": 256},
        {"name": "bezier-65536", "kind": "bezier", "curves": 65536, "threshold": 32, "parent_block": 256},
        {"name": "bezier-262144", "kind": "bezier", "curves": 262144, "threshold": NEVER, "parent_block": 448},
        # triangle counting over a degree-ordered orientation, in the form the benchmark uses
        {"name": "triangles-2e17", "kind": "triangles", "n": 1 << 17, "degree": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bfs", "bfs", "sssp", "sssp", "road", "sssp-multi", "bfs-multi", "batch-bfs", "batch-sssp",
                       "serve", "bezier", "bezier", "bezier", "triangles"])
    if kind in ("bfs", "sssp"):
        graph = rng.choice(["rmat", "rmat", "zipf"])
        n = _log(rng, 1000, 1 << 20)
        return {"kind": kind, "graph": graph, "n": n, "degree": rng.randint(3, 6) if graph == "zipf" else rng.randint(4, 16)}
    if kind == "road":
        return {"kind": rng.choice(["sssp", "bfs"]), "graph": "road", "n": _log(rng, 40, 514) * _log(rng, 40, 514),
                "degree": 6}
    if kind in ("sssp-multi", "bfs-multi"):
        q = rng.randint(2, 16)
        return {"kind": kind, "graph": "rmat", "n": _log(rng, 1000, (1 << 18) * 16 // max(q, 8) // 2), "degree": rng.randint(4, 16),
                "queries": q}
    if kind in ("batch-bfs", "batch-sssp"):
        lo = rng.uniform(8.0, 12.0)
        return {"kind": kind, "count": rng.randint(4, 40), "log2_lo": lo, "log2_hi": rng.uniform(lo + 1.0, 16.5)}
    if kind == "serve":
        return {"kind": kind, "n": _log(rng, 1000, 1 << 16), "degree": rng.randint(4, 16), "queries": rng.randint(4, 48)}
    if kind == "bezier":
        form = rng.choice([(32, 256), (NEVER, 448), (NEVER, 512)])
        return {"kind": kind, "curves": _log(rng, 1, 262144), "threshold": form[0], "parent_block": form[1]}
    return {"kind": "triangles", "n": _log(rng, 500, 1 << 17), "degree": rng.randint(4, 16)}


# ------------------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _csr(n, src, dst):
    key = (src * n + dst).sort().values
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    return row_ptr.to(torch.int32), (key % n).to(torch.int32)


def _rmat_edges(n, m, gen):
    """R-MAT (.57, .19, .19, .05) at scale ceil(log2 n); self-loops and endpoints >= n are redrawn."""
    scale = max(1, math.ceil(math.log2(n)))
    src = torch.zeros(m, dtype=torch.int64, device=DEV)
    dst = torch.zeros(m, dtype=torch.int64, device=DEV)
    todo = torch.arange(m, device=DEV)
    while todo.numel():
        s = torch.zeros(todo.numel(), dtype=torch.int64, device=DEV)
        d = torch.zeros_like(s)
        for _ in range(scale):
            r = torch.rand(todo.numel(), generator=gen, device=DEV)
            s = 2 * s + (r >= 0.76)
            d = 2 * d + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
        src[todo], dst[todo] = s, d
        todo = todo[(s == d) | (s >= n) | (d >= n)]
    return src, dst


def _rmat(n, degree, gen):
    return _csr(n, *_rmat_edges(n, n * degree, gen))


def _zipf(n, gen):
    """Zipf(2.1) out-degrees on [1, 1024], neighbours uniform over the other vertices."""
    k = torch.arange(1, min(1024, n - 1) + 1, dtype=torch.float64, device=DEV)
    cdf = (k ** -2.1).cumsum(0)
    u = torch.rand(n, generator=gen, device=DEV, dtype=torch.float64) * cdf[-1]
    deg = torch.searchsorted(cdf, u).clamp_(max=k.numel() - 1) + 1
    src = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    dst = torch.randint(0, n - 1, (src.numel(),), generator=gen, device=DEV)
    return _csr(n, src, dst + (dst >= src))


def _road(n, gen):
    """Grid digraph: 4 axis edges and each diagonal with probability 1/2."""
    cols = max(2, int(math.isqrt(n)))
    rows = max(1, n // cols)
    v = torch.arange(rows * cols, device=DEV)
    r, c = v // cols, v % cols
    coin = torch.rand(4, v.numel(), generator=gen, device=DEV) < 0.5
    src, dst = [], []
    for k, (dr, dc) in enumerate([(-1, 0), (1, 0), (0, -1), (0, 1), (-1, -1), (-1, 1), (1, -1), (1, 1)]):
        ok = (r + dr >= 0) & (r + dr < rows) & (c + dc >= 0) & (c + dc < cols)
        if k >= 4:
            ok &= coin[k - 4]
        src.append(v[ok])
        dst.append((v + dr * cols + dc)[ok])
    return _csr(rows * cols, torch.cat(src), torch.cat(dst))


def _oriented(n, degree, gen):
    """The simple undirected graph under an R-MAT draw, each edge from the endpoint of lower
    (degree, id) to the other, out-lists sorted."""
    s, d = _rmat_edges(n, n * degree, gen)
    key = torch.unique(torch.cat([s * n + d, d * n + s]))
    s, d = key // n, key % n
    rank = torch.empty(n, dtype=torch.int64, device=DEV)
    rank[torch.bincount(s, minlength=n).sort(stable=True).indices] = torch.arange(n, device=DEV)
    keep = rank[s] < rank[d]
    return _csr(n, s[keep], d[keep])


def _graph(case, gen):
    """{row_ptr, col, w, n, csr} of a weighted digraph on the GPU."""
    if case["graph"] == "rmat":
        row_ptr, col = _rmat(case["n"], case["degree"], gen)
    elif case["graph"] == "zipf":
        row_ptr, col = _zipf(case["n"], gen)
    else:
        row_ptr, col = _road(case["n"], gen)
    w = torch.randint(1, 256, (col.numel(),), generator=gen, device=DEV, dtype=torch.int32)
    return {"row_ptr": row_ptr, "col": col, "w": w, "n": row_ptr.numel() - 1, "csr": npb.make_csr(row_ptr, col, w)}


def _sources(g, count, seed):
    """Vertices with out-edges, drawn uniformly."""
    some = torch.nonzero(g["row_ptr"][1:] > g["row_ptr"][:-1]).reshape(-1).cpu().numpy()
    return some[np.random.RandomState(seed % (1 << 32)).randint(0, len(some), count)].astype(np.int32)


def _instances(case):
    """(n, degree) of a batch's instances: n spread over [2^log2_lo, 2^log2_hi] by its logarithm, large
    and small ones mixed, degrees in [8, 32]."""
    count, lo, hi = case["count"], case["log2_lo"], case["log2_hi"]
    step = next(k for k in (7, 5, 3, 1) if math.gcd(k, count) == 1)
    return [(int(2.0 ** (lo + (hi - lo) * (i * step % count + 0.5) / count)), 8 + i * 11 % 25) for i in range(count)]


def _capacity(case):
    """Points a program sets aside: a random curve has about 95, at most 4096."""
    return 110 * case["curves"] + 8192


def _curves(case, gen):
    k = torch.randint(0, 1 << 24, (case["curves"], 3, 2), generator=gen, device=DEV)
    return k.to(torch.float32) * 2.0 ** -24


def _point_counts(ctrl):
    """Points of each curve: clamp(ceil(64 sqrt(|P0 - 2 P1 + P2| / |P2 - P0|)), 4, 4096) in 64 bits."""
    p = ctrl.double()
    second, chord = p[:, 0] - 2 * p[:, 1] + p[:, 2], p[:, 2] - p[:, 0]
    a = torch.sqrt(second[:, 0] * second[:, 0] + second[:, 1] * second[:, 1])
    b = torch.sqrt(chord[:, 0] * chord[:, 0] + chord[:, 1] * chord[:, 1])
    t = torch.ceil(torch.sqrt(a / b) * 64).nan_to_num(nan=4.0, posinf=4096.0)
    return t.clamp(4, 4096).to(torch.int64)


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    ctx = _context()
    cfg = npb.np_config_default()
    s = {"kind": kind, "ctx": ctx.handle, "cfg": cfg}
    if kind in ("bfs", "sssp"):
        s["graph"] = _graph(case, gen)
        s["out"] = torch.empty(s["graph"]["n"], dtype=torch.int32, device=DEV)
    elif kind in ("bfs-multi", "sssp-multi"):
        s["graph"] = _graph(case, gen)
        s["sources"] = _sources(s["graph"], case["queries"], seed)
        s["ld"] = npb.multi_stride(s["graph"]["n"])
        s["out"] = torch.empty(case["queries"], s["ld"], dtype=torch.int32, device=DEV)
    elif kind in ("batch-bfs", "batch-sssp"):
        graphs = [_graph({"graph": "rmat", "n": n, "degree": degree}, gen) for n, degree in _instances(case)]
        what = npb.NP_BATCH_BFS if kind == "batch-bfs" else npb.NP_BATCH_SSSP
        handle = npb.np_batch_create(ctx.handle, [g["csr"] for g in graphs], [0] * len(graphs), what, cfg)
        s["batch"] = _Kept(handle, npb.np_batch_destroy)
        _, total = npb.np_batch_layout(handle, len(graphs))
        s["out"] = torch.empty(total, dtype=torch.int32, device=DEV)
    elif kind == "serve":
        s["graphs"] = [_graph({"graph": "rmat", "n": n, "degree": case["degree"]}, gen)
                       for n in (case["n"], max(500, case["n"] // 3))]
        torch.cuda.synchronize()
        handle = npb.np_server_create(ctx.handle, [g["csr"] for g in s["graphs"]], memory_budget=2 << 30, max_slots=16)
        s["server"] = _Kept(handle, npb.np_server_destroy)
        per = [max(1, case["queries"] // 4)] * 4
        s["sources"] = [_sources(s["graphs"][i // 2], per[i], seed + i).tolist() for i in range(4)]
        s["out"] = [torch.empty(per[i], s["graphs"][i // 2]["n"], dtype=torch.int32, device=DEV) for i in range(4)]
    elif kind == "bezier":
        s["cfg"] = cfg.replace(threshold=case["threshold"], parent_block=case["parent_block"])
        s["ctrl"] = _curves(case, gen)
        s["cap"] = _capacity(case)
        s["offsets"] = torch.zeros(case["curves"] + 1, dtype=torch.int32, device=DEV)
        s["points"] = torch.zeros(s["cap"], 2, dtype=torch.float32, device=DEV)
    else:
        row_ptr, col = _oriented(case["n"], case["degree"], gen)
        s["cfg"] = cfg.replace(threshold=8, child_block=32, cfactor=1)
        s["graph"] = {"row_ptr": row_ptr, "col": col, "csr": npb.make_csr(row_ptr, col)}
        s["out"] = torch.zeros(1, dtype=torch.int64, device=DEV)
    return s


def run(s):
    kind, ctx, cfg = s["kind"], s["ctx"], s["cfg"]
    if kind == "bfs":
        npb.np_bfs(ctx, s["graph"]["csr"], 0, s["out"], cfg)
    elif kind == "sssp":
        npb.np_sssp(ctx, s["graph"]["csr"], 0, s["out"], cfg)
    elif kind == "bfs-multi":
        npb.np_bfs_multi(ctx, s["graph"]["csr"], s["sources"], s["out"], s["ld"], cfg)
    elif kind == "sssp-multi":
        npb.np_sssp_multi(ctx, s["graph"]["csr"], s["sources"], s["out"], s["ld"], cfg)
    elif kind in ("batch-bfs", "batch-sssp"):
        npb.np_batch_run(s["batch"].handle, s["out"])
    elif kind == "serve":
        sv = s["server"].handle
        for i in range(4):
            for src, out in zip(s["sources"][i], s["out"][i]):
                npb.np_server_submit(sv, i // 2, i % 2, src, out)
        while npb.np_server_step(sv):
            pass
        npb.np_server_finished(sv)
    elif kind == "bezier":
        npb.np_bezier(ctx, s["ctrl"], s["ctrl"].shape[0], s["offsets"], s["points"], s["cap"], cfg)
        return [s["offsets"], s["points"]]
    else:
        npb.np_triangles(ctx, s["graph"]["csr"], s["out"], cfg)
    return s["out"]


# ------------------------------------------------------------------------------ floors

def work(case):
    """Each input read once, each output written once; one addition per relaxed edge, one
    comparison per oriented edge, 12 operations per point (a random curve has about 95)."""
    kind = case["kind"]
    if kind == "bezier":
        nc = case["curves"]
        return {"bytes": 28 * nc + 8 * 95 * nc, "flops": 12 * 95 * nc}
    if kind in ("batch-bfs", "batch-sssp"):
        n = sum(n for n, _ in _instances(case))
        m = sum(n * degree for n, degree in _instances(case))
        return {"bytes": 8 * n + (8 if kind == "batch-sssp" else 4) * m, "flops": m}
    n, m = case["n"], case["n"] * case["degree"]
    if kind == "triangles":
        return {"bytes": 4 * n + 4 * m, "flops": m}
    if kind == "serve":
        n, m = n + max(500, n // 3), (n + max(500, n // 3)) * case["degree"]
        per = max(1, case["queries"] // 4)
        return {"bytes": 4 * n + 8 * m + 2 * per * 4 * n, "flops": 2 * per * m}
    queries = case.get("queries", 1)
    return {"bytes": 4 * n + (8 if kind.startswith("sssp") else 4) * m + 4 * n * queries, "flops": queries * m}


def exact(case, seed):
    """Tessellation points in 64 bits. Levels, distances, offsets and counts are whole numbers:
    they have one right value and no rounding."""
    if case["kind"] != "bezier":
        return None
    ctrl = _curves(case, _generator(seed))
    counts = _point_counts(ctrl)
    p = ctrl.double()
    curve = torch.repeat_interleave(torch.arange(p.shape[0], device=DEV), counts)
    first = counts.cumsum(0) - counts
    t = ((torch.arange(curve.numel(), device=DEV) - first[curve]).double() / (counts[curve] - 1).double())[:, None]
    points = torch.zeros(_capacity(case), 2, dtype=torch.float64, device=DEV)
    points[:curve.numel()] = (1 - t) ** 2 * p[curve, 0] + 2 * (1 - t) * t * p[curve, 1] + t * t * p[curve, 2]
    return [None, points]
