"""What the launches ask of a device follows from the device, not from the one the
constants were chosen on: the sizes of the resident grids, as host functions.
"""
import os
import re
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


@needs_nvcc
def test_solver_grid_fits_the_device(tmp_path):
    """Small systems take one cluster of 16 blocks only where the device holds one; else
    they, like the larger ones, take clusters of 8, no more blocks than fit."""
    for fits, blocks, entries, nodes, grid, cluster, small in _run(tmp_path, r"""
#include <cstdio>
#include "amg.cuh"
int main() {
    for (int fits : {0, 1})
        for (int blocks : {8, 24, 144, 152, 400})
            for (long long e0 : {0ll, 1ll, 40000ll, 40001ll, 6000000ll})
                for (long long n0 : {1ll, 4096ll, 4097ll}) {
                    const bchar::SolveShape s = bchar::solve_shape_of(e0, n0, {blocks, fits != 0});
                    std::printf("%d %d %lld %lld %d %d %d\n", fits, blocks, e0, n0, s.grid, s.cluster, s.small);
                }
}
"""):
        assert small == (fits and entries <= 40000 and nodes <= 4096)
        if small:
            assert (grid, cluster) == (16, 16)
        else:
            assert cluster == 8 and grid % 8 == 0 and 8 <= grid <= min(blocks, 256)


def test_opt_ins_are_not_kept_per_process():
    """A function's attributes are one device's: a flag that outlives the handle would
    leave them unset on the second device that a process uses (and its threads would race on it)."""
    flag = re.compile(r"^\s+static (?!const\b|constexpr\b|__|std::mutex\b)\w[\w<>:\s*]*?(\w+)\s*(\[\w*\])?\s*(=|;|\{\})", re.M)
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            found = [m.group(0).strip() for m in flag.finditer(f.read())]
        if name == "noalloc.cu":  # an address per device, behind a lock
            assert found == ["static double *addr[256] ="]
        else:
            assert not found, (name, found)


@needs_nvcc
def test_shared_memory_of_large_systems_leaves_room_for_l1(tmp_path):
    """Where the finest level's columns and weights (12 bytes an entry) cannot all be in the
    blocks' shared memory, a block asks for less of it."""
    for blocks, entries, smem in _run(tmp_path, r"""
#include <cstdio>
#include "amg.cuh"
int main() {
    for (int blocks : {16, 144, 152})
        for (long long per : {1ll, 10800ll, 15999ll, 16000ll, 16001ll, 700000ll})
            std::printf("%d %lld %zu\n", blocks, per * blocks + (per > 16000), bchar::solve_smem_of(per * blocks + (per > 16000), blocks));
}
"""):
        assert smem == (200 if entries <= 16000 * blocks else 144) * 1024
        assert smem == 144 * 1024 or entries * 12 <= smem * blocks
