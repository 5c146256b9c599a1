"""The rules that choose launch shapes from a lattice's size (csrc/lbm_plan.h), on the host."""
import os
import shutil
import subprocess

import pytest

import paper_1402_2920_gb300 as P

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1402_2920_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "lbm_plan.h"
// reads lines of "nx ny nz", writes the rows of CTAs of each tiled kernel's grid that depend on the lattice
int main()
{
    long long d[3];
    while (std::scanf("%lld %lld %lld", &d[0], &d[1], &d[2]) == 3) {
        const int64_t dims[3] = {d[0], d[1], d[2]};
        const int w = lbm::wide_tiles(dims) ? 64 : 32;
        const int64_t ty = lbm::pair_tile_rows(w);
        std::printf("%d %lld\n", w, (long long)((dims[1] + ty - 1) / ty));
    }
    return 0;
}
"""


def _run(tmp_path, source, text):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(source)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout.split("\n")


def test_grids_of_the_tallest_lattices_fit(tmp_path):
    """Every ny that lbm_create accepts gives a grid of at most 65535 rows, whatever tile nx asks for."""
    ny = (4, 262139, 262140, 262141, 262144, 262145, 524279, 524280)
    dims = [(nx, y, 4) for nx in (4, 32, 34, 60, 64, 66, 128, 130, 160, 192, 256) for y in ny]
    dims = [d for d in dims if P.lbm_footprint_bytes(P.LBM_D3Q59, d, P.LBM_STORE_F32_DEV) > 0]
    assert {d[1] for d in dims} == set(ny)
    out = _run(tmp_path, PROGRAM, "\n".join("%d %d %d" % d for d in dims))
    for d, line in zip(dims, out):
        width, rows = (int(v) for v in line.split())
        assert rows <= 65535, (d, width, rows)
    # ... and the width is that of nx alone up to the last ny whose rows fit
    wide = {d[0]: int(line.split()[0]) for d, line in zip(dims, out) if d[1] == 262140}
    assert wide[34] == wide[64] == wide[128] == wide[256] == 64 and wide[4] == wide[66] == 32


def test_tile_widths_of_the_pairwise_collision(tmp_path):
    """64 wide where that pads nx by at most a fifth more than 32 wide."""
    wide = (34, 62, 64, 98, 100, 128, 130, 160, 192, 256, 288)
    narrow = (4, 32, 66, 90, 96)
    out = _run(tmp_path, PROGRAM, "\n".join("%d 8 8" % nx for nx in wide + narrow))
    got = {nx: int(line.split()[0]) for nx, line in zip(wide + narrow, out)}
    assert all(got[nx] == 64 for nx in wide) and all(got[nx] == 32 for nx in narrow)
