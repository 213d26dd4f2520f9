"""Memory of a layer's build: its scratch goes back to the device, so that what
is sized from the free memory afterwards (a server's result arena, another
library's pool) is not smaller for it."""
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


def test_scratch_returns(api):
    """Some 8 M vertices, whose build takes far more scratch than the 1 GB that may stay reserved for the next one."""
    n, k = 700, 16
    g = dict(x0=0.0, y0=0.0, x1=float(n), y1=float(n), nx=1024, ny=1024)
    ang = 2 * np.pi * torch.arange(k, device="cuda", dtype=torch.float64) / k
    r = 0.2 + 0.25 * torch.rand((n * n, k), device="cuda", dtype=torch.float64)
    cx = torch.arange(n, device="cuda", dtype=torch.float64).repeat(n)[:, None] + 0.5
    cy = torch.arange(n, device="cuda", dtype=torch.float64).repeat_interleave(n)[:, None] + 0.5
    verts = torch.stack([cx + r * torch.cos(ang), cy + r * torch.sin(ang)], 2).reshape(-1, 2).contiguous()
    off = torch.arange(0, n * n * k + 1, k, device="cuda", dtype=torch.int64)
    poly = torch.arange(n * n + 1, device="cuda", dtype=torch.int64)
    torch.cuda.synchronize()
    for _ in range(2):
        before = torch.cuda.mem_get_info()[0]
        with api.pip_layer(verts, off, poly, g):
            pass
        torch.cuda.synchronize()
        assert before - torch.cuda.mem_get_info()[0] <= 1100 << 20
        before = torch.cuda.mem_get_info()[0]
        with api.p2p_layer(verts, off, 0.1, g):
            pass
        torch.cuda.synchronize()
        assert before - torch.cuda.mem_get_info()[0] <= 1100 << 20
