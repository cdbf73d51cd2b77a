"""The loops over small levels (np_config.small_parents) where they can go wrong: for SSSP
the distance window, lists that run full, and the changes to and from the grids; for BFS
the queue and its limits. Levels and distances must match the oracle bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import DevGraph, bfs, sssp
from invariants import csr_from_edges
from paper_2201_02789_gb300 import gen
from paper_2201_02789_gb300 import nestpar as npb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = npb.Context(0)
    yield c
    c.close()


def _road(rows, cols, lo, hi):
    """A grid whose frontier grows past the window's size (and, at 330 x 310, past the frontier limit
    if nothing is deferred)."""
    g = gen.road_grid(rows, cols, seed=9, weights=None)
    g.w = gen.uniform_int(9, gen.S_WEIGHT, 0, g.m, lo, hi).astype(np.uint32)
    return g


def _wide(hubs, degree, seed):
    """0 -> hubs vertices of `degree` children each, all into one pool: wide parents (2048 children or
    more), more of them than one CTA (64) or the cluster (1024) can publish in a round, or none."""
    rng = np.random.default_rng(seed)
    pool = hubs + 1 + rng.integers(0, 4000, size=(hubs, degree))
    src = np.concatenate([np.zeros(hubs, np.int64), np.repeat(np.arange(1, hubs + 1), degree)])
    dst = np.concatenate([np.arange(1, hubs + 1), pool.reshape(-1)])
    order = np.argsort(src, kind="stable")
    n = hubs + 4001
    row_ptr = np.zeros(n + 1, np.int32)
    row_ptr[1:] = np.cumsum(np.bincount(src, minlength=n))
    w = rng.integers(1, 256, size=len(src)).astype(np.uint32)
    return gen.Csr(n, row_ptr, dst[order].astype(np.int32), w)


def _pulse():
    """Few vertices, then 30000, then few again: the grids take over and give back."""
    rng = np.random.default_rng(5)
    edges = [(0, 1), (1, 2)] + [(2, 3 + i) for i in range(30000)]
    edges += [(3 + i, 30003 + int(rng.integers(0, 50))) for i in range(30000)]
    edges += [(30003 + i, 30053 + i % 7) for i in range(50)] + [(30053 + i, 30060) for i in range(7)]
    edges += [(30060 + i, 30061 + i) for i in range(20)]
    rp, col, w = csr_from_edges(30081, edges, [int(x) for x in rng.integers(1, 256, size=len(edges))])
    return gen.Csr(30081, rp, col, w)


GRAPHS = {
    "road-300": lambda: _road(300, 300, 1, 255),
    "road-330x310": lambda: _road(330, 310, 1, 255),
    "road-zero-weights": lambda: _road(120, 130, 0, 3),
    "road-equal-weights": lambda: _road(200, 201, 7, 7),
    "road-large-weights": lambda: _road(230, 220, 1, 4000000),
    "wide-70": lambda: _wide(70, 515, 1),
    "wide-1100": lambda: _wide(1100, 513, 2),
    "wide-3000": lambda: _wide(3000, 520, 3),
    "wide-70x2047": lambda: _wide(70, 2047, 4),
    "wide-70x2048": lambda: _wide(70, 2048, 5),
    "wide-1100x2100": lambda: _wide(1100, 2100, 6),
    "pulse": _pulse,
    "rmat-13007": lambda: gen.rmat(14, 12, seed=21, n=13007, m=13007 * 12),
    "rmat-17001": lambda: gen.rmat(15, 24, seed=22, n=17001, m=17001 * 24),
}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_distances(ctx, name):
    g = GRAPHS[name]()
    dg = DevGraph(g)
    for src in (0, g.n // 2):
        ref = oracle.sssp(g.row_ptr, g.col, g.w, src)
        for kw in ({}, {"small_parents": 300}, {"small_parents": 5, "unroll": 1}, {"sweep_parents": 0, "unroll": 2}):
            d, st = sssp(ctx, dg, src, npb.config("tca", **kw), stats=True)
            np.testing.assert_array_equal(d, ref)
            assert st["error"] == 0 and st["timeouts"] == 0


def _alternating(pairs):
    """Levels of 3 and 60 vertices in turn: with a limit between the two, a while body of two levels
    that starts at a wide one ends before the next wide one, just after a narrow one."""
    g, src = _fan(80 * pairs, [3, 60] * pairs, 11)
    g.w = gen.uniform_int(11, gen.S_WEIGHT, 0, g.m, 1, 255).astype(np.uint32)
    return g, src


@pytest.mark.parametrize("unroll", [2, 3, 5, 8, 11, 15])
def test_levels_left_to_the_grids(ctx, unroll):
    """The loop at a body's end that finds too large a frontier leaves it to the grids as it is,
    whatever the number of levels in the body."""
    g, src = _alternating(100)
    big = GRAPHS["rmat-17001"]()
    for g, src in ((g, src), (big, 0)):
        dg = DevGraph(g)
        ref = oracle.sssp(g.row_ptr, g.col, g.w, src)
        for kw in ({"small_parents": 1}, {"small_parents": 40, "sweep_parents": 0}, {}):
            d, st = sssp(ctx, dg, src, npb.config("tca", unroll=unroll, **kw), stats=True)
            np.testing.assert_array_equal(d, ref)
            assert st["error"] == 0 and st["timeouts"] == 0


def test_several_sources_share_the_window(ctx):
    """Queries of one call share one window, whatever their distances."""
    g = _road(150, 140, 1, 255)
    dg = DevGraph(g)
    sources = [0, g.n - 1, g.n // 2, 139, 77]
    ld = npb.multi_stride(g.n)
    dist = torch.empty(len(sources), ld, dtype=torch.int32, device="cuda:0")
    npb.np_sssp_multi(ctx.handle, dg.csr, sources, dist, ld, npb.config("tca"), stats=True)
    out = dist.cpu().numpy().view(np.uint32)
    for q, s in enumerate(sources):
        np.testing.assert_array_equal(out[q, :g.n], oracle.sssp(g.row_ptr, g.col, g.w, s))


# ---- BFS from its start in one CTA (visited bits in shared memory)

def _fan(n, widths, seed):
    """Levels of the given widths, every vertex of one with edges into the next (some with none,
    some twice to the same vertex); the rest of the n vertices unreached."""
    rng = np.random.default_rng(seed)
    ids = rng.permutation(n)[:1 + sum(widths)]
    src, dst, at = [ids[:0]], [ids[:0]], 1
    prev = ids[:1]
    for w in widths:
        cur = ids[at:at + w]
        at += w
        src += [prev[rng.integers(0, max(1, len(prev) * 3 // 4), w)], prev[:1], prev[:1]]
        dst += [cur, cur[:1], cur[:1]]
        prev = cur
    src, dst = np.concatenate(src), np.concatenate(dst)
    order = np.argsort(src, kind="stable")
    row_ptr = np.zeros(n + 1, np.int32)
    row_ptr[1:] = np.cumsum(np.bincount(src, minlength=n))
    return gen.Csr(n, row_ptr, dst[order].astype(np.int32)), int(ids[0])


FANS = {
    "words": (129, [3, 40, 80]),
    "parents-8192": (40000, [3, 8192, 8193, 40, 8000, 5]),
    "children-16384": (60000, [16384, 100, 16385, 7]),
    "queue": (1 << 20, [4, 5500, 8000, 12000, 20, 7000, 9]),      # 128 KB of bits: 5632 queued parents
    "no-bits": ((1 << 20) + 1, [4, 5500, 8000, 12000, 20, 7000, 9]),
    "isolated": (7, []),
}


@pytest.mark.parametrize("name", list(FANS))
def test_bfs_first_levels(ctx, name):
    n, widths = FANS[name]
    g, src = _fan(n, widths, len(name))
    dg = DevGraph(g)
    ref = oracle.bfs(g.row_ptr, g.col, src)
    for kw in ({}, {"small_parents": 100}, {"sweep_parents": 0, "unroll": 1}):
        lv, st = bfs(ctx, dg, src, npb.config("tca", **kw), stats=True)
        np.testing.assert_array_equal(lv, ref)
        assert st["error"] == 0 and st["parents"] == (ref >= 0).sum()
        assert st["levels"] == ref.max() + 1 and st["pushes"] == (ref > 0).sum()
        assert st["items"] == np.diff(g.row_ptr)[ref >= 0].sum()


@pytest.mark.parametrize("rows,cols", [(40, 41), (300, 310)])
def test_bfs_road(ctx, rows, cols):
    g = gen.road_grid(rows, cols, seed=4, weights=None)
    dg = DevGraph(g)
    for src in (0, g.n // 2):
        np.testing.assert_array_equal(bfs(ctx, dg, src, npb.config("tca")), oracle.bfs(g.row_ptr, g.col, src))


@pytest.mark.parametrize("unroll", [1, 2, 3, 5, 8, 11, 15])
def test_bfs_levels_left_to_the_grids(ctx, unroll):
    """As test_levels_left_to_the_grids, for the one-CTA loop at the end of a body."""
    g, src = _alternating(100)
    big = GRAPHS["rmat-17001"]()
    for g, src in ((g, src), (big, 0)):
        dg = DevGraph(g)
        ref = oracle.bfs(g.row_ptr, g.col, src)
        for kw in ({"small_parents": 8}, {"small_parents": 40, "sweep_parents": 0}, {}):
            lv, st = bfs(ctx, dg, src, npb.config("tca", unroll=unroll, **kw), stats=True)
            np.testing.assert_array_equal(lv, ref)
            assert st["error"] == 0 and st["levels"] == ref.max() + 1
