"""The tessellation's count and point grids at the edges of their tiles (256 curves, 64 per
point CTA, 1024 tiles summed by the point CTAs themselves, one grid for both up to 512 curves),
with parent subsets and a capacity
that falls inside a tile. Offsets exact; points |g - r| <= 1e-5 max(|r|, 1) as everywhere
(three exact integer weights times products rounded twice: below 1e-6)."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import DevGraph, bezier
from invariants import bezier_tolerance_ok
from paper_2201_02789_gb300 import gen
from paper_2201_02789_gb300 import nestpar as npb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = npb.Context(0)
    yield c
    c.close()


def _few_points(n):
    """n curves of 4 to 14 points (nearly straight), every 1000th a random one."""
    ctrl = gen.bezier_curves(n, seed=51)
    mid = (ctrl[:, 0] + ctrl[:, 2]) * np.float32(0.5)
    flat = mid + (ctrl[:, 1] - mid) * np.float32(1e-4)
    out = ctrl.copy()
    out[:, 1] = flat
    out[::1000] = ctrl[::1000]
    return np.ascontiguousarray(out)


@pytest.mark.parametrize("nc", [1, 8, 63, 64, 65, 255, 256, 257, 511, 512, 513, 4097, 262144, 262145, 300001])
def test_tile_edges(ctx, nc):
    ctrl = _few_points(nc) if nc > 10000 else gen.bezier_curves(nc, seed=52)
    ref_off, ref_pts = oracle.bezier(ctrl)
    for kw in ({}, {"threshold": npb.INT32_MAX, "parent_grid": 3}):
        status, off, pts, st = bezier(ctx, ctrl, npb.config("tca", **kw), cap=int(ref_off[-1]))
        assert status == npb.NP_OK and st["error"] == 0
        np.testing.assert_array_equal(off, ref_off)
        ok, worst = bezier_tolerance_ok(pts, ref_pts)
        assert ok, worst
        assert st["items"] == ref_off[-1] and st["parents"] == nc
        big = int((np.diff(ref_off) >= 32).sum()) if not kw else 0
        assert st["launch_parents"] == big and st["serial_parents"] == nc - big


@pytest.mark.parametrize("nc", [301, 500, 700, 262500])
def test_capacity_inside_a_tile(ctx, nc):
    ctrl = _few_points(nc)
    ref_off, ref_pts = oracle.bezier(ctrl)
    fit = nc - 300                       # the last curve that fits, in the middle of a tile
    cap = int(ref_off[fit + 1]) + 1
    status, off, pts, st = bezier(ctx, ctrl, npb.config("tca"), cap=cap, check=False)
    assert status == npb.NP_ERR_CAPACITY
    np.testing.assert_array_equal(off, ref_off)
    inside = int(np.searchsorted(ref_off, cap, side="right") - 1)
    ok, worst = bezier_tolerance_ok(pts[:ref_off[inside]], ref_pts[:ref_off[inside]])
    assert ok, worst
    assert np.isnan(pts[ref_off[inside]:cap]).all()      # a curve that does not fit writes nothing
    assert st["items"] == ref_off[inside]


WIDE_FORMS = {
    "points": {}, "count-grid-3": dict(threshold=npb.INT32_MAX, parent_grid=3), "nodp": dict(variant=npb.NP_VARIANT_NODP),
    "nodp-cta": dict(variant=npb.NP_VARIANT_NODP, granularity="none"), "cta": dict(serial=npb.NP_SERIAL_BLOCK),
    "packed": dict(serial=npb.NP_SERIAL_PACKED), "none": dict(granularity="none"), "warp": dict(granularity="warp"),
    "block": dict(granularity="block"), "grid_device": dict(granularity="grid_device", scan=npb.NP_SCAN_LOOKBACK),
}


def _closed(n):
    """n curves that end where they begin: 4096 points each."""
    ctrl = np.zeros((n, 3, 2), np.float32)
    ctrl[:, 1] = [0.5, 0.25]
    return torch.from_numpy(ctrl).cuda()


@pytest.mark.parametrize("nc", [(1 << 19) + 77, (1 << 20) + 300], ids=["above-2^31", "above-2^32"])
@pytest.mark.parametrize("form", list(WIDE_FORMS))
def test_totals_beyond_32_bits(ctx, form, nc):
    """More points than an int32 offset can number: the curves that end within the capacity are
    written and nothing else, offsets beyond INT32_MAX hold INT32_MAX."""
    c_d, cap, guard = _closed(nc), 10000, 1 << 22
    off = torch.full((nc + 1,), -7, dtype=torch.int32, device="cuda:0")
    pts = torch.full((guard + cap + guard, 2), float("nan"), dtype=torch.float32, device="cuda:0")
    status, st = npb.np_bezier(ctx.handle, c_d, nc, off, pts[guard:], cap, npb.config("tca", **WIDE_FORMS[form]),
                               stats=True, check=False)
    assert status == npb.NP_ERR_CAPACITY
    want = np.minimum(np.arange(nc + 1, dtype=np.int64) * 4096, npb.INT32_MAX)
    np.testing.assert_array_equal(off.cpu().numpy(), want)
    written = ~torch.isnan(pts[:, 0])
    assert written[guard:guard + 8192].all() and int(written.sum()) == 8192
    assert st["items"] == 8192 and st["parents"] == nc


def test_capacity_beyond_32_bits(ctx):
    """A buffer of more than 2^31 points: what ends beyond INT32_MAX is skipped all the same."""
    nc = (1 << 19) + 2
    c_d, cap = _closed(nc), nc * 4096
    off = torch.full((nc + 1,), -7, dtype=torch.int32, device="cuda:0")
    pts = torch.full((cap, 2), float("nan"), dtype=torch.float32, device="cuda:0")
    status, st = npb.np_bezier(ctx.handle, c_d, nc, off, pts, cap, npb.config("tca"), stats=True, check=False)
    assert status == npb.NP_ERR_CAPACITY
    fit = (npb.INT32_MAX // 4096) * 4096
    assert torch.isfinite(pts[fit - 4096:fit]).all() and torch.isnan(pts[fit:]).all()
    assert st["items"] == fit


def test_parent_subset_with_padding(ctx):
    ctrl = gen.bezier_curves(600, seed=53)
    ids = np.arange(599, -1, -1, dtype=np.int32)[:520].copy()
    ids[[0, 255, 256, 300, 519]] = -1
    counts = np.array([oracle.bezier_count(ctrl[i]) if i >= 0 else 0 for i in ids])
    dev = "cuda:0"
    c_d, id_d = torch.from_numpy(ctrl).to(dev), torch.from_numpy(ids).to(dev)
    off = torch.full((len(ids) + 1,), -7, dtype=torch.int32, device=dev)
    pts = torch.empty((int(counts.sum()), 2), dtype=torch.float32, device=dev)
    body = npb.np_body(kind=npb.NP_BODY_BEZIER_EVAL, ctrl=c_d.data_ptr(), offsets=off.data_ptr(),
                       points=pts.data_ptr(), cap=int(counts.sum()))
    _, st = npb.np_run_nested(ctx.handle, npb.np_parents(id_d.data_ptr(), len(ids)), npb.NP_COUNT_BEZIER, None, body,
                              npb.config("tca"), stats=True)
    o, p = off.cpu().numpy(), pts.cpu().numpy()
    first = np.concatenate([[0], np.cumsum(counts)])
    assert st["parents"] == (ids >= 0).sum() and o[-1] == first[-1]
    np.testing.assert_array_equal(o[:-1][ids >= 0], first[:-1][ids >= 0])
    assert (o[:-1][ids < 0] == -7).all()                 # padding holds no parent: its offset is not written
    for k in np.flatnonzero(ids >= 0)[::7]:
        for j in (0, counts[k] - 1):
            assert bezier_tolerance_ok(p[first[k] + j], oracle.bezier_point(ctrl[ids[k]], counts[k], j))[0]


@pytest.mark.parametrize("count", [1, 64, 65, 300, 512])
def test_padded_parents_in_one_grid(ctx, count):
    ctrl = gen.bezier_curves(600, seed=54)
    ids = np.random.default_rng(count).permutation(600)[:count].astype(np.int32)
    ids[::5] = -1
    keep = ids >= 0
    n_of = np.array([oracle.bezier_count(ctrl[i]) if i >= 0 else 0 for i in ids])
    first = np.concatenate([[0], np.cumsum(n_of)])
    c_d, id_d = torch.from_numpy(ctrl).cuda(), torch.from_numpy(ids).cuda()
    for cap in (int(first[-1]), int(first[-1]) // 2):
        off = torch.full((count + 1,), -7, dtype=torch.int32, device="cuda:0")
        pts = torch.full((int(first[-1]) + 1, 2), float("nan"), dtype=torch.float32, device="cuda:0")
        body = npb.np_body(kind=npb.NP_BODY_BEZIER_EVAL, ctrl=c_d.data_ptr(), offsets=off.data_ptr(),
                           points=pts.data_ptr(), cap=cap)
        status, st = npb.np_run_nested(ctx.handle, npb.np_parents(id_d.data_ptr(), count), npb.NP_COUNT_BEZIER, None,
                                       body, npb.config("tca"), stats=True, check=False)
        assert status == (npb.NP_OK if first[-1] <= cap else npb.NP_ERR_CAPACITY)
        o, p = off.cpu().numpy(), pts.cpu().numpy()
        np.testing.assert_array_equal(o[:-1][keep], first[:-1][keep])
        assert (o[:-1][~keep] == -7).all() and o[-1] == first[-1]
        fits = keep & (first[1:] <= cap)
        assert st["parents"] == keep.sum() and st["items"] == n_of[fits].sum()
        assert st["launch_parents"] == (n_of[fits] >= 32).sum()
        for k in np.flatnonzero(keep):
            row = p[first[k]:first[k + 1]]
            if fits[k]:
                ref = np.array([oracle.bezier_point(ctrl[ids[k]], n_of[k], j) for j in range(n_of[k])])
                assert bezier_tolerance_ok(row, ref)[0]
            else:
                assert np.isnan(row).all()


def test_refused_under_capture(ctx):
    """A context's workspace may be freed by a later call, so its passes are not captured."""
    ctrl = torch.from_numpy(gen.bezier_curves(700, seed=55)).cuda()
    off = torch.empty(701, dtype=torch.int32, device="cuda:0")
    pts = torch.empty(200000, 2, dtype=torch.float32, device="cuda:0")
    npb.np_bezier(ctx.handle, ctrl, 700, off, pts, 200000)
    dg, count = DevGraph(gen.rmat(8, 4, seed=3)), torch.zeros(1, dtype=torch.int64, device="cuda:0")
    npb.np_triangles(ctx.handle, dg.csr, count)
    torch.cuda.synchronize()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        off.zero_()
        assert npb.np_bezier(ctx.handle, ctrl, 700, off, pts, 200000, check=False) == npb.NP_ERR_CUDA
        assert npb.np_bezier(ctx.handle, ctrl, 700, off, pts, 200000, npb.config("nodp"),
                             check=False) == npb.NP_ERR_CUDA
        assert npb.np_triangles(ctx.handle, dg.csr, count, check=False) == npb.NP_ERR_CUDA


@pytest.mark.parametrize("gran", ["none", "warp", "block", "multiblock", "grid_device"])
def test_after_device_launched_children(ctx, gran):
    """A pass whose grid may be scheduled early still waits for the children that the pass before it
    launched from the device: both write the same points."""
    a, b = (torch.from_numpy(gen.bezier_curves(n, seed=n)).cuda() for n in (3000, 300))
    off = torch.empty(3001, dtype=torch.int32, device="cuda:0")
    pts = torch.empty(600000, 2, dtype=torch.float32, device="cuda:0")
    npb.np_bezier(ctx.handle, b, 300, off, pts, 600000)
    total = int(off[300].item())
    ref = pts[:total].clone()
    for _ in range(5):
        npb.np_bezier(ctx.handle, a, 3000, off, pts, 600000, npb.config("tca", granularity=gran, threshold=0))
        npb.np_bezier(ctx.handle, b, 300, off, pts, 600000)
        assert int(off[300].item()) == total and torch.equal(pts[:total], ref)


def _scaled_curves(n, seed):
    """Curves of all magnitudes down to the smallest subnormal: whole curves scaled, x and y scaled
    apart, single coordinates; every fourth one closed (4096 points)."""
    rng = np.random.default_rng(seed)
    u = rng.uniform(-1, 1, (n, 3, 2))
    e = rng.integers(-149, 3, (n, 1, 1)).astype(np.float64)
    e = np.where(np.arange(n)[:, None, None] % 3 == 1, rng.integers(-149, 3, (n, 1, 2)), e)
    e = np.where(np.arange(n)[:, None, None] % 3 == 2, rng.integers(-149, 3, (n, 3, 2)), e)
    ctrl = (u * 2.0 ** e).astype(np.float32)
    ctrl[::4, 2] = ctrl[::4, 0]
    return np.ascontiguousarray(ctrl)


@pytest.mark.parametrize("nc", [300, 3000])
@pytest.mark.parametrize("kw", [{}, {"threshold": npb.INT32_MAX, "parent_grid": 3}])
def test_points_of_any_magnitude(ctx, nc, kw):
    """Each coordinate to 9 units of 2^-24 of the sum of its three terms' magnitudes and 4 halves
    of the smallest subnormal. The longest chain: the reciprocal, t and u by it (two roundings each,
    in a product of two of them), that product, its product with the coordinate and two sums: 8; one
    more for second-order terms. A rounding to a subnormal is half of 2^-149, three products and
    the sums at most four of them."""
    ctrl = _scaled_curves(nc, seed=56)
    ref_off = oracle.bezier_offsets(ctrl)
    status, off, pts, _ = bezier(ctx, ctrl, npb.config("tca", **kw), cap=int(ref_off[-1]))
    assert status == npb.NP_OK
    np.testing.assert_array_equal(off, ref_off)
    n_of = np.diff(ref_off)
    curve = np.repeat(np.arange(nc), n_of)
    j = (np.arange(ref_off[-1]) - ref_off[:-1][curve]).astype(np.float64)
    t, u = j / (n_of[curve] - 1), (n_of[curve] - 1 - j) / (n_of[curve] - 1)
    terms = np.stack([u * u, 2 * u * t, t * t], 1)[:, :, None] * ctrl.astype(np.float64)[curve]
    bound = 9 * 2.0 ** -24 * np.abs(terms).sum(1) + 4 * 2.0 ** -150
    worst = (np.abs(pts.astype(np.float64) - terms.sum(1)) / bound).max()
    assert worst <= 1.0, worst
