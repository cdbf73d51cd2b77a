"""The parent grid's tiles of 32 parents, taken by a fixed stride with the next tiles loaded
ahead (thresholds up to 128) or from a ticket: edges of tiles, one CTA for all of them, padded
frontiers. Levels and distances must match the oracle bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import DevGraph, bfs, sssp
from paper_2201_02789_gb300 import gen
from paper_2201_02789_gb300 import nestpar as npb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = npb.Context(0)
    yield c
    c.close()


def _graph(width, seed):
    """0 -> `width` vertices of 0 to 300 children each, with weights."""
    rng = np.random.default_rng(seed)
    n = 2 * width + 200
    deg = rng.integers(0, 8, n)
    deg[1:1 + width:7] = rng.integers(100, 300, len(deg[1:1 + width:7]))
    deg[0] = width
    row_ptr = np.zeros(n + 1, np.int32)
    row_ptr[1:] = np.cumsum(deg)
    col = rng.integers(0, n, int(row_ptr[-1])).astype(np.int32)
    col[:width] = np.arange(1, width + 1)
    return gen.Csr(n, row_ptr, col, rng.integers(0, 256, len(col)).astype(np.uint32))


@pytest.mark.parametrize("threshold", [0, 128, 129])
@pytest.mark.parametrize("width", [1, 31, 32, 33, 257, 9001])
def test_solves(ctx, width, threshold):
    g = _graph(width, width + threshold)
    dg = DevGraph(g)
    level, dist = oracle.bfs(g.row_ptr, g.col, 0), oracle.sssp(g.row_ptr, g.col, g.w, 0)
    for grid in (0, 1, 3):
        for sweep in (0, 1):
            cfg = npb.config("tca", threshold=threshold, parent_grid=grid, sweep_parents=sweep, small_parents=0)
            np.testing.assert_array_equal(bfs(ctx, dg, 0, cfg), level)
            np.testing.assert_array_equal(sssp(ctx, dg, 0, cfg), dist)


@pytest.mark.parametrize("threshold", [128, 129])
@pytest.mark.parametrize("count", [1, 31, 32, 33, 64, 255, 256, 257, 5000])
def test_padded_parents(ctx, count, threshold):
    """One pass over a parent list in which every third slot is padding (-1)."""
    g = _graph(6000, count)
    dg = DevGraph(g)
    ids = np.random.default_rng(count).permutation(g.n)[:count].astype(np.int32)
    level0 = np.full(g.n, -1, np.int32)
    level0[ids] = 0
    want = level0.copy()
    want_next = np.sort(oracle.bfs_expand(g.row_ptr, g.col, np.delete(ids, np.s_[::3]), 0, want))
    ids[::3] = -1
    for grid in (0, 1):
        level, cur = torch.from_numpy(level0).cuda(), torch.from_numpy(ids).cuda()
        nxt = torch.empty(g.n, dtype=torch.int32, device="cuda:0")
        cnt = torch.zeros(1, dtype=torch.int32, device="cuda:0")
        body = npb.np_body(kind=npb.NP_BODY_BFS_VISIT, next_level=1, level=level.data_ptr(), next=nxt.data_ptr(),
                           next_count=cnt.data_ptr())
        npb.np_run_nested(ctx.handle, npb.np_parents(cur.data_ptr(), count), npb.NP_COUNT_CSR_DEGREE, dg.csr, body,
                          npb.config("tca", threshold=threshold, parent_grid=grid))
        np.testing.assert_array_equal(level.cpu().numpy(), want)
        np.testing.assert_array_equal(np.sort(nxt[:int(cnt.item())].cpu().numpy()), want_next)
