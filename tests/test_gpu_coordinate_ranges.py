"""Grids whose coordinates or cells leave the FP32 range: cells and row lists
must be the FP64 rule's, the joins those of the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (lower corner, cell): coordinates beyond the largest FP32 number, also with
# cells below it, and cells so small that FP32 subnormals count, with a cell
# boundary between zero and the smallest normal number (2^-126 = 1.2e-38)
RANGES = [(0.0, 1e40), (0.0, 2e38), (-3e41, 1e40), (-37.995e-36, 1e-36)]


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0802_gb300 import api as A
    from paper_1403_0802_gb300 import build
    build.build()
    return A


def grid(x0, cell, n=64):
    return dict(x0=x0, y0=x0, x1=x0 + n * cell, y1=x0 + n * cell, nx=n, ny=n)


def special_points(rng, g, cell):
    """Uniform points, cell boundaries and their neighbours, tiny values, and
    values far outside of any range."""
    u = g["x0"] + rng.uniform(-0.1, 1.1, (6_000, 2)) * (g["x1"] - g["x0"])
    tiny = u[:1_000].copy()
    tiny[:500, 0] = rng.uniform(-1.5e-38, 1.5e-38, 500)
    tiny[500:, 1] = rng.uniform(-1.5e-38, 1.5e-38, 500)
    k = g["x0"] + np.arange(g["nx"] + 1) * cell
    k = np.concatenate([k, np.nextafter(k, np.inf), np.nextafter(k, -np.inf)])
    far = np.array([1e60, -1e60, 1e300, 3.5e38, -3.5e38, np.inf, -np.inf, np.nan])
    edge = np.concatenate([k, far])
    mid = rng.uniform(g["x0"], g["x1"], len(edge))
    return np.concatenate([u, tiny, np.stack([edge, mid], 1), np.stack([mid, edge], 1)])


@pytest.mark.parametrize("x0,cell", RANGES)
def test_cells(api, x0, cell):
    g = grid(x0, cell)
    pts = special_points(np.random.default_rng(1), g, cell)
    with np.errstate(all="ignore"):
        w = (g["x1"] - g["x0"]) / 64
        c = np.floor((pts - x0) / w)
        inside = (c >= 0).all(1) & (c < 64).all(1)
    want = (c[:, 1] * 64 + c[:, 0])
    start, perm = (t.cpu().numpy() for t in api.bucket_points(torch.as_tensor(pts, device="cuda"), g))
    assert start[-1] == inside.sum()
    got = np.full(len(pts), -1.0)
    got[perm[:start[-1]]] = np.repeat(np.arange(64 * 64), np.diff(start))
    np.testing.assert_array_equal(got, np.where(inside, want, -1))


@pytest.mark.parametrize("x0,cell", RANGES)
def test_polygons(api, oracle, x0, cell):
    rng = np.random.default_rng(5)
    g = grid(x0, cell)

    def star(cx, cy, r0, r1, n):
        ang = 2 * np.pi * (np.arange(n) + rng.uniform(0, 0.9, n)) / n
        r = rng.uniform(r0, r1, n)
        return np.stack([cx + r * np.cos(ang), cy + r * np.sin(ang)], 1)

    rings = [x0 + cell * r for r in (star(16, 20, 4, 12, 40), star(44, 40, 6, 17, 7), star(44, 40, 2, 9, 300),
                                     star(37.5, 38.5, 2, 5, 90))]
    verts = np.concatenate(rings)
    off = np.concatenate([[0], np.cumsum([len(r) for r in rings])]).astype(np.int64)
    poly = np.arange(len(rings) + 1, dtype=np.int64)
    pts = np.concatenate([special_points(rng, g, cell), verts, 0.5 * (verts + np.roll(verts, -1, 0))])
    ref = oracle.pip_join(g, pts, verts, off, poly)
    assert (ref >= 0).any() and (ref < 0).any()
    dev = torch.as_tensor(pts, device="cuda")
    with api.pip_layer(verts, off, poly, g) as layer:
        for form in ("fp64",) if max(abs(g["x0"]), abs(g["x1"])) > 1e30 else ("fp64", "fp32x"):
            np.testing.assert_array_equal(api.pip_join(layer, dev, form=form).cpu().numpy(), ref)


@pytest.mark.parametrize("x0,cell", RANGES)
def test_polylines(api, oracle, x0, cell):
    rng = np.random.default_rng(7)
    g = grid(x0, cell)
    verts = x0 + rng.uniform(3, 61, (120, 2)) * cell
    off = np.arange(0, 121, 4, dtype=np.int64)
    pts = special_points(rng, g, cell)
    D = 3.0 * cell
    rid, rd, d1, d2 = oracle.p2p_join(g, pts, verts, off, D)
    with np.errstate(invalid="ignore"):      # inf - inf: no polyline at all
        clear = ~((np.abs(d2 - d1) <= 1e-9 * cell) | (np.abs(d1 - D) <= 1e-9 * D))
    dev = torch.as_tensor(pts, device="cuda")
    with api.p2p_layer(verts, off, D, g) as layer:
        for ppi in (0, 128):                 # straight over the points, and bucketed
            gid, gd = (t.cpu().numpy() for t in api.p2p_join(layer, dev, form="fp64", pts_per_item=ppi))
            np.testing.assert_array_equal(gid[clear], rid[clear])
            hit = (gid >= 0) & (rid >= 0)
            assert hit.any()
            # both FP64, up to the order of operations: relative to the distance
            # and to the coordinates that it is taken from
            tol = 1e-12 * np.maximum(rd[hit], cell) + 4e-16 * abs(x0)
            assert np.all(np.abs(gd[hit] - rd[hit]) <= tol)


@pytest.mark.parametrize("scale", [1e-30, 1e-9, 1.0, 1e17, 1e27])
def test_fp32x_squares_out_of_range(api, oracle, scale):
    """FP32X where the squares of distances overflow or underflow FP32: every
    point within D of a polyline is found, none beyond it is."""
    rng = np.random.default_rng(2)
    verts = rng.uniform(20, 230, (90, 2)) * scale
    off = np.arange(0, 91, 3, dtype=np.int64)
    g = dict(x0=0.0, y0=0.0, x1=256.0 * scale, y1=256.0 * scale, nx=32, ny=32)
    pts = rng.uniform(-5, 260, (3_000, 2)) * scale
    dev = torch.as_tensor(pts, device="cuda")
    far = 256 * 2 ** 0.5 * scale
    for D in (12.0 * scale, 150.0 * scale):
        rid, rd, d1, d2 = oracle.p2p_join(g, pts, verts, off, D)
        # the distance bound of FP32X (E = 64 u M, u = 2^-24, M at most twice the extent) is below 1e-5 of the extent
        with np.errstate(invalid="ignore"):
            clear = ~((np.abs(d2 - d1) <= 1e-5 * far) | (np.abs(d1 - D) <= 1e-5 * far))
        with api.p2p_layer(verts, off, D, g) as layer:
            got = [api.p2p_join(layer, dev, form="fp32x", pts_per_item=ppi) for ppi in (0, 128)]
            got.append(api.p2p_join(layer, dev, form="fp32x", window=D))
            oid, od = torch.empty_like(got[0][0]), torch.empty_like(got[0][1])
            got.append(api.p2p_join_noalloc(layer, dev, oid, od, form="fp32x"))
            out = (torch.empty_like(oid), torch.empty_like(od))
            with api.Engine(max_points=len(pts), max_requests=1, form="fp32x") as eng:
                s = torch.cuda.Stream()
                eng.round([(layer, dev, *out)], s)
                s.synchronize()
            got.append(out)
            torch.cuda.synchronize()
        for gid, gd in got:
            gid, gd = gid.cpu().numpy(), gd.cpu().numpy()
            np.testing.assert_array_equal(gid[clear], rid[clear])
            hit = (gid >= 0) & (rid >= 0)
            assert hit.sum() > 100
            assert np.all(np.abs(gd[hit] - rd[hit]) <= 1e-5 * far)


@pytest.mark.parametrize("x0,cell,n", [(0.0, 1.0, 64), (4.5e6, 0.37, 64), (-8e6, 250.0, 2048), (-1e5, 1e-3, 1024),
                                       (0.0, 1e40, 64), (-37.995e-36, 1e-36, 64), (0.0, 1e-38, 64), (1e-38, 1e-39, 64)])
def test_points_outside(api, oracle, x0, cell, n):
    """Points on, next to and far from the grid's ends: a polygon that covers the grid holds those inside alone."""
    g = grid(x0, cell, n)
    rng = np.random.default_rng(11)
    verts = np.array([[g["x0"], g["y0"]], [g["x1"], g["y0"]], [g["x1"], g["y1"]], [g["x0"], g["y1"]]])
    off, poly = np.array([0, 4], np.int64), np.array([0, 1], np.int64)
    end = np.repeat([g["x0"], g["x1"]], 400)
    near = [end, np.nextafter(end, np.inf), np.nextafter(end, -np.inf),
            end + rng.uniform(-1, 1, end.size) * 10.0 ** rng.uniform(-9, 2, end.size) * cell,
            end * (1 + rng.uniform(-1, 1, end.size) * 10.0 ** rng.uniform(-16, -5, end.size)),
            rng.uniform(-1, 1, end.size) * 10.0 ** rng.uniform(-40, 300, end.size)]
    edge = np.concatenate(near + [np.array([np.inf, -np.inf, np.nan, 0.0, -0.0])])
    mid = rng.uniform(g["x0"], g["x1"], edge.size)
    pts = np.concatenate([np.stack([edge, mid], 1), np.stack([mid, edge], 1), np.stack([edge, edge[::-1]], 1)])
    ref = oracle.pip_join(g, pts, verts, off, poly)
    assert (ref >= 0).any() and (ref < 0).any()
    with api.pip_layer(verts, off, poly, g) as layer:
        got = api.pip_join(layer, torch.as_tensor(pts, device="cuda"), form="fp64").cpu().numpy()
    np.testing.assert_array_equal(got, ref)
