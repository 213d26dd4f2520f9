"""Launch shapes that a kernel's fixed-size state depends on, for GPUs and parts
of GPUs of any number of SMs (host arithmetic only; no GPU)."""
import os
import subprocess

from paper_1403_0802_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "sj_internal.cuh"
using namespace sj;
int main() {
    // a block of the direct polyline join takes runs of DIRECT_WARPS points, one run in every `blocks`
    for (int sms = 1; sms <= 160; ++sms)
        for (int n = 1; n <= P2P_DIRECT_FP32X; n += n < 70 || n > P2P_DIRECT_FP32X - 200 ? 1 : 37) {
            const int blocks = p2p_direct_blocks(n, sms), runs = (n + DIRECT_WARPS - 1) / DIRECT_WARPS;
            const int most = (runs + blocks - 1) / blocks * DIRECT_WARPS;
            if (blocks < 1 || most > DIRECT_OPEN) {
                std::printf("%d points on %d SMs: %d blocks of up to %d points\n", n, sms, blocks, most);
                return 1;
            }
        }
    return 0;
}
"""


def test_direct_join_blocks(tmp_path):
    src, exe = tmp_path / "shapes.cu", tmp_path / "shapes"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
