"""What the launches ask of a device follows from the device, not from the one the
constants were chosen on: the sizes of the resident grids, as host functions.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_05834_gb300", "csrc")
NVCC = os.environ.get("NVCC", "nvcc")
needs_nvcc = pytest.mark.skipif(shutil.which(NVCC) is None, reason="needs nvcc (host code only)")


def _run(tmp_path, source):
    src, exe = tmp_path / "p.cu", tmp_path / "p"
    src.write_text(source)
    r = subprocess.run([NVCC, "-std=c++17", "-arch=sm_103a", "--expt-relaxed-constexpr", "-I", CSRC,
                        "-I", os.path.join(CSRC, "..", "..", "include"), "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return [[int(v) for v in line.split()] for line in subprocess.check_output([str(exe)], text=True).splitlines()]


@needs_nvcc
def test_interior_point_grid_fits_the_device(tmp_path):
    """A cooperative grid larger than what is resident at once is refused: with 148,
    28 or 1 blocks the grid is no larger, from one cell to 10^9."""
    for resident, cells, grid in _run(tmp_path, r"""
#include <cstdio>
#include "ip.cuh"
int main() {
    for (int resident : {1, 28, 148, 152, 160, 400})
        for (long long nc : {1ll, 64ll, 65ll, 9472ll, 9473ll, 1000000000ll})
            std::printf("%d %lld %d\n", resident, nc, bchar::ip_grid(nc, resident));
}
"""):
        assert 1 <= grid <= resident
        assert grid <= max(1, (cells + 63) // 64)
        if resident <= 152:
            assert grid == min(resident, (cells + 63) // 64)
