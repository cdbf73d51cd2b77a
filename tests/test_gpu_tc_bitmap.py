"""Triangle counting's child grid with adjacency bitmaps: list lengths around the 32- and
128-entry runs, records longer than a chunk of edges, every CTA size its bitmap takes, and the
change to the intersection per thread above the largest bitmap. Counts are exact."""
import threading

import numpy as np
import pytest
import torch

from paper_2201_02789_gb300 import nestpar as npb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = npb.Context(0)
    yield c
    c.close()


def _count(ctx, n, lists, **kw):
    """Triangles of the DAG with out-lists {u: sorted ids}, through np_triangles."""
    deg = np.zeros(n + 1, np.int64)
    for u, l in lists.items():
        deg[u + 1] = len(l)
    row_ptr = torch.from_numpy(np.cumsum(deg).astype(np.int32)).cuda()
    col = torch.from_numpy(np.concatenate([np.asarray(lists[u], np.int32) for u in sorted(lists)])).cuda()
    out = torch.zeros(1, dtype=torch.int64, device="cuda:0")
    npb.np_triangles(ctx.handle, npb.make_csr(row_ptr, col), out, npb.config("tca", threshold=1, **kw), stats=True)
    return int(out.item())


def _expected(lists):
    s = {u: set(map(int, l)) for u, l in lists.items()}
    return sum(len(s[u] & s.get(v, set())) for u in s for v in s[u])


@pytest.mark.parametrize("kw", [dict(child_block=32, cfactor=1), dict(child_block=64, cfactor=4),
                                dict(child_block=1024, cfactor=16), dict(child_block=32, cfactor=2, serial=2)],
                         ids=["cb32", "cb64x4", "cb1024x16", "block"])
def test_run_lengths(ctx, kw):
    """Two kinds of lists over 700 ids: short and long heads against bodies of 1..260 entries."""
    rng = np.random.default_rng(3)
    n, lists = 3000, {}
    for i, k in enumerate([1, 2, 31, 32, 33, 63, 64, 65, 95, 96, 127, 128, 129, 159, 160, 191, 255, 256, 257, 260]):
        lists[200 + i] = np.sort(rng.choice(np.arange(1000, 1700), k, replace=False))
    bodies = np.arange(200, 220)
    for u in range(100):
        own = rng.choice(np.arange(1000, 1700), int(rng.integers(1, 300)), replace=False)
        lists[u] = np.sort(np.concatenate([rng.choice(bodies, int(rng.integers(1, 20)), replace=False), own]))
    assert _count(ctx, n, lists, **kw) == _expected(lists)


@pytest.mark.parametrize("n", [1000, 1024, 131072, 131073, 300000, 600000, 1000001, 1638400, 1638401])
def test_bitmap_sizes(ctx, n):
    """Ids over the whole range, among them the first and the last, and one list of 700 edges
    (several chunks) into lists that meet it."""
    rng = np.random.default_rng(n)
    ids = np.unique(np.concatenate([[n - 1, n - 2, n // 2], rng.integers(n // 4, n, 900)]))
    mids = np.arange(1, 1 + min(700, n // 8))
    lists = {0: np.concatenate([mids, ids[-200:]])}
    for v in mids[::3]:
        lists[int(v)] = np.sort(rng.choice(ids, int(rng.integers(1, min(150, len(ids)))), replace=False))
    assert _count(ctx, n, lists, child_block=32, cfactor=1) == _expected(lists)


def test_two_contexts_in_two_threads():
    """Bitmaps of 16 KB and 200 KB counted at the same time through contexts of their own: neither
    call changes what the other's launch may take."""
    jobs = []
    for n in (131072, 1638400):
        rng = np.random.default_rng(n)
        ids = np.unique(rng.integers(n // 4, n, 900))
        lists = {0: np.concatenate([np.arange(1, 300), ids[-200:]])}
        for v in range(1, 300, 3):
            lists[v] = np.sort(rng.choice(ids, int(rng.integers(40, 150)), replace=False))
        deg = np.zeros(n + 1, np.int64)
        for u, l in lists.items():
            deg[u + 1] = len(l)
        row_ptr = torch.from_numpy(np.cumsum(deg).astype(np.int32)).cuda()
        col = torch.from_numpy(np.concatenate([np.asarray(lists[u], np.int32) for u in sorted(lists)])).cuda()
        jobs.append((npb.make_csr(row_ptr, col), _expected(lists), row_ptr, col))
    torch.cuda.synchronize()
    start, errors = threading.Barrier(len(jobs)), []

    def work(csr, want):
        try:
            with npb.Context(0) as c:
                s = torch.cuda.Stream()
                out = torch.zeros(400, dtype=torch.int64, device="cuda:0")
                torch.cuda.synchronize()
                start.wait(timeout=60)
                for i in range(len(out)):
                    npb.np_triangles(c.handle, csr, out[i:], npb.config("tca", threshold=1), stream=s)
                s.synchronize()
                assert (out == want).all()
        except Exception as e:   # (reported by the main thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=j[:2]) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
