"""Points of a polygon join that wait for the general refinement are kept in
lists of their own: outputs that requests of a round share do not reach other
requests, and calls that need the lists' scratch report when it is refused."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRID = dict(x0=0.0, y0=0.0, x1=64.0, y1=64.0, nx=4, ny=4)


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0802_gb300 import _lib as L
    from paper_1403_0802_gb300 import api as A
    from paper_1403_0802_gb300 import build
    build.build()
    yield A, L
    L.lib().sj_fault_inject(0, 0, 0)


@pytest.fixture(scope="module")
def rough():
    """One polygon of 4,000 edges over 16 cells: every list is searched, so every point of its cells waits."""
    rng = np.random.default_rng(4)
    ang = 2 * np.pi * np.arange(4_000) / 4_000
    r = rng.uniform(20, 31, 4_000)
    verts = np.stack([32 + r * np.cos(ang), 32 + r * np.sin(ang)], 1)
    return verts, np.array([0, 4_000], np.int64), np.array([0, 1], np.int64)


def test_shared_outputs_in_a_round(lib, rough, oracle):
    A, _ = lib
    n = 300_000   # three requests: several tiles per warp, in different requests
    rng = np.random.default_rng(8)
    a, c = rng.uniform(0, 64, (n, 2)), rng.uniform(0, 64, (n, 2))
    want_a, want_c = (oracle.pip_join(GRID, p, *rough) for p in (a, c))
    with A.pip_layer(*rough, GRID) as layer, A.Engine(max_points=3 * n, max_requests=3, form="fp32x") as eng:
        pa, pc = (torch.as_tensor(p, device="cuda") for p in (a, c))
        out_a, out_c = (torch.full((n,), 7, dtype=torch.int32, device="cuda") for _ in range(2))
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        for _ in range(3):   # the same points twice, into the same output
            eng.round([(layer, pa, out_a, None), (layer, pa, out_a, None), (layer, pc, out_c, None)], s)
        s.synchronize()
    np.testing.assert_array_equal(out_c.cpu().numpy(), want_c)
    np.testing.assert_array_equal(out_a.cpu().numpy(), want_a)


@pytest.mark.parametrize("n", [155_649, 622_591, 622_592, 1_245_184, 1_245_185, 3_000_001])
def test_scratch_refused(lib, rough, oracle, n):
    """Around the sizes (on 152 SMs) where a warp has a second tile, tiles hold two points per lane and the lists
    need scratch."""
    A, L = lib
    pts = np.random.default_rng(n).uniform(-1, 65, (n, 2))
    want = oracle.pip_join(GRID, pts, *rough)
    p = torch.as_tensor(pts, device="cuda")
    out = torch.full((n,), 7, dtype=torch.int32, device="cuda")
    needs = n > 8 * 32 * 32 * torch.cuda.get_device_properties(0).multi_processor_count
    with A.pip_layer(*rough, GRID) as layer:
        L.lib().sj_fault_inject(1, 0, 1)   # the next allocation is refused
        try:
            if needs:
                with pytest.raises(L.SJError) as e:
                    A.pip_join(layer, p, out)
                assert e.value.status == L.SJ_ERR_OOM
                torch.cuda.synchronize()
                assert bool((out == 7).all())
        finally:
            L.lib().sj_fault_inject(0, 0, 0)
        A.pip_join(layer, p, out)
        np.testing.assert_array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("n", [1, 3, 4, 5, 1_003, 19_456, 19_457, 38_912, 38_913, 77_824, 77_825, 155_648])
def test_small_tiles(lib, rough, oracle, n):
    """Small calls take tiles of 4, 8, 16 or 32 points (the sizes where they change on 152 SMs); every point waits."""
    A, _ = lib
    pts = np.random.default_rng(n).uniform(-1, 65, (n, 2))
    out = torch.full((n + 1,), 7, dtype=torch.int32, device="cuda")
    with A.pip_layer(*rough, GRID) as layer:
        A.pip_join(layer, torch.as_tensor(pts, device="cuda"), out[:n], form="fp32x")
        st = layer.stats()
    got = out.cpu().numpy()
    want = oracle.pip_join(GRID, pts, *rough)
    np.testing.assert_array_equal(got[:n], want)
    assert got[n] == 7 and st["hits"] == (want >= 0).sum()


@pytest.mark.parametrize("most", [1, 1_003, 19_457, 155_649, 1_300_000])
def test_small_rounds(lib, rough, oracle, most):
    """Rounds of an engine for at most `most` points, from one point to all of them, in two requests: tiles of 4 to
    32 points on one grid (every point waits; the largest engine has its lists in scratch)."""
    A, _ = lib
    pts = np.random.default_rng(most).uniform(-1, 65, (most, 2))
    want = oracle.pip_join(GRID, pts, *rough)
    p = torch.as_tensor(pts, device="cuda")
    with A.pip_layer(*rough, GRID) as layer, A.Engine(max_points=most, max_requests=2, form="fp32x") as eng:
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        for n in sorted({1, min(most, 2), min(most, 129), (most + 3) // 4, (most + 1) // 2, most}):
            out = torch.full((n + 1,), 7, dtype=torch.int32, device="cuda")
            s.wait_stream(torch.cuda.current_stream())
            k = n // 3
            eng.round([(layer, p[:k], out[:k], None), (layer, p[k:n], out[k:n], None)], s)
            s.synchronize()
            got = out.cpu().numpy()
            np.testing.assert_array_equal(got[:n], want[:n])
            assert got[n] == 7
