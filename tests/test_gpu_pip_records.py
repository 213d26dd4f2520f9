"""The PIP join's cell records at the sizes where their handling changes: groups
of 32 candidates, inline and separate candidate ids, lists scanned, searched or
ordered by a block, many flips, edges shared by two and three polygons, cells
that the FP32 estimate leaves open, coordinates beyond the FP32 range.  Ids are
compared with the oracle bit for bit (no tolerance), in both forms, for points
on vertices, on edges and on cell boundaries besides uniform ones, and with the
search threshold lowered (the sub-cell flag)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0802_gb300 import api as A
    from paper_1403_0802_gb300 import build
    build.build()
    return A


def layer_of(rings):
    sizes = [len(r) for r in rings]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    return np.ascontiguousarray(np.concatenate(rings), np.float64), off, np.arange(len(rings) + 1, dtype=np.int64)


def points_of(rng, verts, g, n=20_000):
    lo, hi = np.array([g["x0"], g["y0"]]), np.array([g["x1"], g["y1"]])
    nxt = np.roll(verts, -1, 0)
    bx = g["x0"] + np.arange(g["nx"] + 1) * ((g["x1"] - g["x0"]) / g["nx"])
    on_cells = np.stack([rng.choice(bx, 500), rng.uniform(lo[1], hi[1], 500)], 1)
    ty = np.stack([rng.uniform(lo[0], hi[0], len(verts)), verts[:, 1]], 1)       # ties with vertices in y
    return np.concatenate([rng.uniform(lo - 0.01 * (hi - lo), hi + 0.01 * (hi - lo), (n, 2)), verts,
                           0.5 * (verts + nxt), ty, on_cells, [[np.nan, lo[1]], [np.inf, hi[1]]]])


def check(api, oracle, rings, g, seed):
    verts, off, poly = layer_of(rings)
    pts = points_of(np.random.default_rng(seed), verts, g)
    ref = oracle.pip_join(g, pts, verts, off, poly)
    assert (ref >= 0).any() and (ref < 0).any()
    with api.pip_layer(verts, off, poly, g) as layer:
        dev = torch.as_tensor(pts, device="cuda")
        for form in ("fp64", "fp32x"):
            for sub in (None, True):
                got = api.pip_join(layer, dev, form=form, subcell=sub).cpu().numpy()
                np.testing.assert_array_equal(got, ref)
        st = layer.stats()
        assert st["hits"] == 4 * (ref >= 0).sum()
        out = torch.full((len(pts),), 7, dtype=torch.int32, device="cuda")
        with api.Engine(max_points=len(pts), max_requests=3, form="fp64") as eng:   # as three requests
            s = torch.cuda.Stream()
            a, b = len(pts) // 3, len(pts) // 2
            eng.round([(layer, dev[i:j].contiguous(), out[i:j], None) for i, j in ((0, a), (a, b), (b, len(pts)))], s)
            s.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy(), ref)


def star(rng, cx, cy, r0, r1, n):
    ang = 2 * np.pi * (np.arange(n) + rng.uniform(0, 0.9, n)) / n
    r = rng.uniform(r0, r1, n)
    return np.stack([cx + r * np.cos(ang), cy + r * np.sin(ang)], 1)


GRID = dict(x0=0.0, y0=0.0, x1=64.0, y1=64.0, nx=4, ny=4)


@pytest.mark.parametrize("k", [1, 3, 4, 31, 32, 33, 64, 70])
def test_stacked_candidates(api, oracle, k):
    """k overlapping polygons in every cell, a full-cover one among them."""
    rng = np.random.default_rng(k)
    rings = [star(rng, 32 + rng.uniform(-4, 4), 32 + rng.uniform(-4, 4), 4, 27, 9) for _ in range(k)]
    rings.insert(k // 2, np.array([[1.0, 1.0], [63.0, 1.0], [63.0, 30.0], [1.0, 30.0]]))
    check(api, oracle, rings, GRID, k)


@pytest.mark.parametrize("m", [8, 9, 15, 16, 17, 31, 32, 33, 255, 256, 257, 700, 3000])
@pytest.mark.parametrize("vertical", [True, False])
def test_list_lengths(api, oracle, m, vertical):
    """A zigzag side of m edges inside one row or column of cells, across a
    cell boundary (so that edges and flips both number about m), shared by two
    polygons; the left one is given twice (a third copy of every edge)."""
    t = np.linspace(17.0, 31.0, m + 1)
    z = 32.0 + np.where(np.arange(m + 1) % 2, 1.5, -1.25) * (1 + 0.1 * np.sin(np.arange(m + 1)))
    zig = np.stack([z, t], 1) if vertical else np.stack([t, z], 1)
    if vertical:
        left = np.concatenate([[[20.0, 17.0]], zig, [[20.0, 31.0]]])
        right = np.concatenate([[[44.0, 31.0]], zig[::-1], [[44.0, 17.0]]])
    else:
        left = np.concatenate([zig, [[31.0, 20.0]], [[17.0, 20.0]]])
        right = np.concatenate([zig[::-1], [[17.0, 44.0]], [[31.0, 44.0]]])
    check(api, oracle, [right, left, left.copy(), np.array([[40.0, 40.0], [60.0, 40.0], [50.0, 60.0]])], GRID, m)


@pytest.mark.parametrize("shift,cell", [((4.5e6, 5.3e6), 0.37), ((0.0, 0.0), 1e29), ((0.0, 0.0), 1e-36)])
def test_coordinate_ranges(api, oracle, shift, cell):
    """Cells far smaller than the FP32 spacing of their coordinates (no cell is
    certain in FP32), coordinates beyond 1e30 and near the smallest floats."""
    rng = np.random.default_rng(5)
    g = dict(x0=shift[0], y0=shift[1], x1=shift[0] + 64 * cell, y1=shift[1] + 64 * cell, nx=64, ny=64)
    rings = [star(rng, 16.0, 20.0, 4, 12, 40), star(rng, 44.0, 40.0, 6, 17, 7), star(rng, 44.0, 40.0, 2, 9, 300)]
    rings = [np.asarray(shift) + r * cell for r in rings]
    check_form = "fp64"
    verts, off, poly = layer_of(rings)
    pts = points_of(rng, verts, g, 5_000)
    ref = oracle.pip_join(g, pts, verts, off, poly)
    assert (ref >= 0).any() and (ref < 0).any()
    with api.pip_layer(verts, off, poly, g) as layer:
        got = api.pip_join(layer, torch.as_tensor(pts, device="cuda"), form=check_form).cpu().numpy()
    np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 128, 129, 622_591, 622_592, 622_593])
def test_point_counts(api, oracle, n):
    """Calls around a warp, a tile and the size where tiles hold two points per lane."""
    rng = np.random.default_rng(n)
    rings = [star(rng, 8 + 16 * i, 8 + 16 * j, 3, 7.9, 12) for j in range(4) for i in range(4)]
    verts, off, poly = layer_of(rings)
    g = dict(GRID, nx=32, ny=32)
    pts = rng.uniform(-1.0, 65.0, (n, 2))
    ref = oracle.pip_join(g, pts, verts, off, poly)
    with api.pip_layer(verts, off, poly, g) as layer:
        out = torch.full((n + 1,), 7, dtype=torch.int32, device="cuda")[1:]   # any 4-byte alignment
        got = api.pip_join(layer, torch.as_tensor(pts, device="cuda"), out, form="fp32x").cpu().numpy()
    np.testing.assert_array_equal(got, ref)


def test_sub_cells(api, oracle):
    """Cells cut by few edges, whose sub-cells without an edge answer from the
    cell table: stars, a rectangle and a comb with horizontal and vertical sides
    on and off the cell and sub-cell lines, a polygon with a hole, dense points
    around the sub-cell lines."""
    rng = np.random.default_rng(3)
    g = dict(x0=0.0, y0=0.0, x1=64.0, y1=64.0, nx=8, ny=8)
    rings = [star(rng, 14, 14, 5, 12, 7), star(rng, 46, 14, 5, 12, 11),
             np.array([[3.0, 34.0], [27.0, 34.0], [27.0, 49.5], [3.0, 49.5]]),
             np.array([[33.0, 33.3], [61.0, 33.3], [61.0, 60.0], [54.0, 60.0], [54.0, 41.0], [47.0, 41.0],
                       [47.0, 60.0], [33.0, 60.0]])]
    hole = star(rng, 14, 14, 1, 3, 5)
    verts = np.concatenate([rings[0], hole] + rings[1:])
    off = np.concatenate([[0], np.cumsum([len(rings[0]), len(hole)] + [len(r) for r in rings[1:]])]).astype(np.int64)
    poly = np.array([0, 2, 3, 4, 5], np.int64)
    line = np.repeat(np.arange(0, 64, 2.0), 200)
    jit = rng.normal(0, 1e-4, line.size)
    pts = np.concatenate([rng.uniform(0, 64, (200_000, 2)), np.stack([line + jit, rng.uniform(0, 64, line.size)], 1),
                          np.stack([rng.uniform(0, 64, line.size), line + jit], 1), points_of(rng, verts, g)])
    ref = oracle.pip_join(g, pts, verts, off, poly)
    with api.pip_layer(verts, off, poly, g) as layer:
        got = api.pip_join(layer, torch.as_tensor(pts, device="cuda"), form="fp32x").cpu().numpy()
        st = layer.stats()
    np.testing.assert_array_equal(got, ref)
    # more points are answered without an edge test than those of the cells that no edge's box meets
    nxt = np.arange(1, len(verts) + 1)
    nxt[off[1:] - 1] = off[:-1]
    lo, hi = np.minimum(verts, verts[nxt]), np.maximum(verts, verts[nxt])
    free = np.ones((8, 8), bool)
    for (ax, ay), (bx, by) in zip((lo / 8).astype(int), (hi / 8).astype(int)):
        free[ay:by + 1, ax:bx + 1] = False
    inside = np.isfinite(pts).all(1) & (pts >= 0).all(1) & (pts < 64).all(1)
    cell = (pts[inside] / 8).astype(int)
    assert st["resolved"] > free[cell[:, 1], cell[:, 0]].sum()
