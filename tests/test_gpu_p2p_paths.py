"""The polyline join's paths against one another and the oracle.

Small calls go straight over the points, larger ones bucket them; the FP64 form
decides in FP32 which segments need FP64.  A call that shapes its work items
(pts_per_item) always buckets, so the same points give both paths: ids and
distances must be the same bits (FP32X too, as long as no cell holds more points
than an item, whose certificate is then that of the cell's points), and meet the
oracle by the bar of tests/parity.py."""
import numpy as np
import pytest

from paper_1403_0802_gb300 import synth
from parity import P2PRef

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FORMS = ("fp64", "fp32x")


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0802_gb300 import api as A
    from paper_1403_0802_gb300 import build
    build.build()
    return A


def both_paths(api, layer, pts, form, window=None):
    p = torch.as_tensor(pts, device="cuda")
    a = api.p2p_join(layer, p, form=form, window=window)
    b = api.p2p_join(layer, p, form=form, window=window, pts_per_item=128)
    torch.testing.assert_close(a[0], b[0], rtol=0, atol=0)
    torch.testing.assert_close(a[1], b[1], rtol=0, atol=0)
    return a[0].cpu().numpy(), a[1].cpu().numpy()


@pytest.fixture(scope="module")
def walks():
    return synth.p2p_walks(n_points=140_000, n_lines=60_000)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("n", [1, 7, 8, 9, 1_003, 9_727, 9_729, 32_768, 32_769, 131_072, 131_073])
def test_point_counts(api, oracle, walks, form, n):
    L = walks.polylines
    ref = P2PRef(oracle, walks.grid, L.verts, L.line_off, walks.D)
    with api.p2p_layer(L.verts, L.line_off, walks.D, walks.grid) as layer:
        pts = walks.points[:n].copy()
        pts[::97] += 1e5                     # outside the grid
        pts[5::501, 1] = np.nan
        gid, gd = both_paths(api, layer, pts, form)
        ok = ~np.isnan(pts).any(1)
        ref.check(np.ascontiguousarray(pts[ok]), gid[ok], gd[ok], form)
        assert (gid[~ok] == -1).all() and np.isinf(gd[~ok]).all()
        st = layer.stats()
        assert st["hits"] == 2 * (gid >= 0).sum()
        if n <= 32_769:
            both_paths(api, layer, pts, form, window=31.25)
            oid = torch.full((n,), 7, dtype=torch.int32, device="cuda")
            od = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
            api.p2p_join_noalloc(layer, torch.as_tensor(pts, device="cuda"), oid, od, form=form)
            torch.cuda.synchronize()
            np.testing.assert_array_equal(oid.cpu().numpy(), gid)


@pytest.mark.parametrize("form", FORMS)
def test_near_ties(api, oracle, form):
    """Points within a few millimetres of the middle of two parallel lines: the
    certificate decides most of them by its magnitude, which depends on the
    work item, and three lines through one vertex leave the FP64 form with
    more than two segments."""
    rng = np.random.default_rng(9)
    lines, pts = [], []
    for k in range(300):
        x, y = 100.0 * rng.integers(4, 60, 2) + rng.uniform(0, 60, 2)
        if k % 3 == 2:                       # a star of three lines: equal distances to the shared vertex
            lines += [[(x, y), (x + 20 * np.cos(t), y + 20 * np.sin(t))] for t in (0.1, 0.9, 1.7)]
            pts += [(x - r, y - 0.7 * r) for r in rng.uniform(0, 15, 20)]
        else:
            lines += [[(x, y), (x + 30.0, y)], [(x, y + 20.0), (x + 30.0, y + 20.0)]]
            pts += [(x + 30.0 * rng.random(), y + 10.0 + rng.normal(0, 1e-3)) for _ in range(20)]
    verts = np.concatenate([np.asarray(l, np.float64) for l in lines])
    off = np.arange(0, 2 * len(lines) + 1, 2, dtype=np.int64)
    pts = np.asarray(pts, np.float64)
    g = dict(x0=0.0, y0=0.0, x1=6400.0, y1=6400.0, nx=32, ny=32)
    ref = P2PRef(oracle, g, verts, off, 40.0)
    with api.p2p_layer(verts, off, 40.0, g) as layer:
        gid, gd = both_paths(api, layer, pts, form)
        assert layer.stats()["fallbacks"] > 100
    ref.check(pts, gid, gd, form)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("lines", [1, 31, 32, 33, 127, 128, 129, 400])
def test_list_lengths(api, oracle, form, lines):
    """Lists of about `lines` segments (one, full and several staging areas),
    with one-vertex polylines and duplicates among them, a window that covers
    the grid, one point per cell and many."""
    rng = np.random.default_rng(lines)
    segs = rng.uniform(10, 246, (lines, 2, 2))
    segs[::7, 1] = segs[::7, 0]              # zero-length
    if lines > 2:
        segs[2] = segs[1]
    verts, off = segs.reshape(-1, 2), np.arange(0, 2 * lines + 1, 2, dtype=np.int64)
    g = dict(x0=0.0, y0=0.0, x1=256.0, y1=256.0, nx=4, ny=4)
    ref = P2PRef(oracle, g, verts, off, 400.0)
    with api.p2p_layer(verts, off, 400.0, g) as layer:
        for n in (3, 1_500):
            pts = np.concatenate([rng.uniform(0, 256, (n, 2)), verts[:50]])
            gid, gd = both_paths(api, layer, pts, form)
            ref.check(pts, gid, gd, form)


@pytest.mark.parametrize("scale,x0", [(1e-9, 0.0), (1e17, 0.0), (1e28, 0.0), (1.0, 4.5e6)])
def test_fp64_coordinate_ranges(api, oracle, scale, x0):
    """Where the FP32 bound has no meaning every point is redone in FP64; grids
    whose coordinates are large against a cell."""
    rng = np.random.default_rng(2)
    verts = x0 + rng.uniform(20, 230, (90, 2)) * scale
    off = np.arange(0, 91, 3, dtype=np.int64)
    g = dict(x0=x0, y0=x0, x1=x0 + 256.0 * scale, y1=x0 + 256.0 * scale, nx=32, ny=32)
    pts = x0 + rng.uniform(-5, 260, (3_000, 2)) * scale
    D = 12.0 * scale
    rid, rd, d1, d2 = oracle.p2p_join(g, pts, verts, off, D)
    with api.p2p_layer(verts, off, D, g) as layer:
        gid, gd = both_paths(api, layer, pts, "fp64")
    with np.errstate(invalid="ignore"):      # inf - inf: no polyline at all
        clear = (np.abs(d2 - d1) > 1e-9 * np.maximum(d1, scale)) & (np.abs(d1 - D) > 1e-9 * D)
    np.testing.assert_array_equal(gid[clear], rid[clear])
    hit = (gid >= 0) & (rid >= 0)
    assert hit.any()
    assert np.all(np.abs(gd[hit] - rd[hit]) <= 1e-12 * np.maximum(rd[hit], scale) + 4e-16 * abs(x0))


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("copies", [2, 3, 15, 16, 17, 31, 32, 33, 70])
def test_coincident_lines(api, oracle, form, copies):
    """Routes that share their streets: every line given `copies` times, so that no point has a single nearest one.
    The points of a warp's FP64 queue hold 2 to 32 segments each, more than 32 leave it; one point and many."""
    rng = np.random.default_rng(copies)
    one = rng.uniform(5, 251, (12, 3, 2))
    verts = np.concatenate([one] * copies).reshape(-1, 2)
    off = np.arange(0, 3 * 12 * copies + 1, 3, dtype=np.int64)
    g = dict(x0=0.0, y0=0.0, x1=256.0, y1=256.0, nx=4, ny=4)
    ref = P2PRef(oracle, g, verts, off, 90.0)
    with api.p2p_layer(verts, off, 90.0, g) as layer:
        for n in (1, 33, 40_000):
            pts = rng.uniform(-5, 261, (n, 2))
            gid, gd = both_paths(api, layer, pts, form)
            ref.check(pts, gid, gd, form)
            assert (gid < 12).all()          # of equal distances the smallest id


@pytest.mark.parametrize("form", FORMS)
def test_few_and_many_coincident_lines(api, oracle, form):
    """Lines given 3 times beside lines given 40 times: a warp takes points that fit its FP64 queue and points that
    leave it in turn, in the same places of shared memory."""
    rng = np.random.default_rng(6)
    one = rng.uniform(5, 251, (24, 3, 2))
    times = np.where(np.arange(24) % 2, 3, 40)
    verts = np.repeat(one, times, axis=0).reshape(-1, 2)
    off = np.arange(0, 3 * times.sum() + 1, 3, dtype=np.int64)
    g = dict(x0=0.0, y0=0.0, x1=256.0, y1=256.0, nx=4, ny=4)
    ref = P2PRef(oracle, g, verts, off, 90.0)
    first = np.concatenate([[0], np.cumsum(times)[:-1]])
    with api.p2p_layer(verts, off, 90.0, g) as layer:
        for n in (40, 40_000, 140_000):
            pts = rng.uniform(-5, 261, (n, 2))
            gid, gd = both_paths(api, layer, pts, form)
            ref.check(pts, gid, gd, form)
            assert np.isin(gid[gid >= 0], first).all()   # of equal distances the smallest id


def test_dense_cells_fp32x(api, oracle):
    """A cell with more points than a work item holds: the direct path certifies each point with all of the call's
    points of its cell, bucketing with those of its item.  Ids are the same; where the distances are not, one is the
    FP32 and the other the FP64 distance, each within the oracle's bound."""
    rng = np.random.default_rng(13)
    segs = rng.uniform(10, 246, (60, 2, 2))
    segs[1::2] = segs[::2] + rng.uniform(1e-3, 3e-3, (30, 1, 1))   # near-ties, which the item can decide
    verts, off = segs.reshape(-1, 2), np.arange(0, 121, 2, dtype=np.int64)
    g = dict(x0=0.0, y0=0.0, x1=256.0, y1=256.0, nx=4, ny=4)
    pts = rng.uniform(0, 256, (32_768, 2))
    ref = P2PRef(oracle, g, verts, off, 400.0)
    r = ref.join(pts)
    with api.p2p_layer(verts, off, 400.0, g) as layer:
        p = torch.as_tensor(pts, device="cuda")
        a, b = api.p2p_join(layer, p, form="fp32x"), api.p2p_join(layer, p, form="fp32x", pts_per_item=128)
        torch.testing.assert_close(a[0], b[0], rtol=0, atol=0)
        for gid, gd in (a, b):
            ref.check(pts, gid.cpu().numpy(), gd.cpu().numpy(), "fp32x", ref=r)
