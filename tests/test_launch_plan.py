"""The rules that choose launch shapes from a lattice's size (csrc/lbm_plan.h), on the host."""
import os
import shutil
import subprocess

import pytest

import paper_1402_2920_gb300 as P

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1402_2920_gb300", "csrc")

ROWS = r"""
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
    out = _run(tmp_path, ROWS, "\n".join("%d %d %d" % d for d in dims))
    for d, line in zip(dims, out):
        width, rows = (int(v) for v in line.split())
        assert rows <= 65535, (d, width, rows)
    # ... and the width is that of nx alone up to the last ny whose rows fit
    wide = {d[0]: int(line.split()[0]) for d, line in zip(dims, out) if d[1] == 262140}
    assert wide[34] == wide[64] == wide[128] == wide[256] == 64 and wide[4] == wide[66] == 32


KEYS = r"""
#include <cstdio>
#include <cstdlib>
#include "lbm_plan.h"
// reads lines of "lattice nx ny nz storage precision gamma", writes batch keys
int main()
{
    long long l, d[3], st, pr;
    double gamma;
    while (std::scanf("%lld %lld %lld %lld %lld %lld %lf", &l, &d[0], &d[1], &d[2], &st, &pr, &gamma) == 7) {
        const int64_t dims[3] = {d[0], d[1], d[2]};
        lbm_params p{};
        p.storage = int(st);
        p.usolve_precision = int(pr);
        p.gamma = gamma;
        std::printf("%d\n", lbm::batch_key(int(l), dims, p));
    }
    return 0;
}
"""


def test_simulations_that_run_the_same_kernels_batch_together(tmp_path):
    """Lattices of one size class (2^14 to 2^16 sites): one key, unless the collision on pairs of sites tells them
    apart."""
    two = [(96 + 32 * k, 128, 1) for k in (1, 2, 3, 4)] + [(129, 131, 1), (161, 130, 1)]
    three = [(34, 32, 32), (32, 32, 33), (33, 32, 32), (48, 30, 30)]
    stores = [P.LBM_STORE_F32, P.LBM_STORE_F32_DEV, P.LBM_STORE_F16_DEV, P.LBM_STORE_BF16_DEV, P.LBM_STORE_F64,
              P.LBM_STORE_F32_LOC, P.LBM_STORE_F16_LOC, P.LBM_STORE_BF16_LOC]
    sets = [(lat, dims, st, pr, g) for lat, dims in ((P.LBM_D2Q21, two), (P.LBM_D3Q59, three)) for st in stores
            for pr in (P.LBM_USOLVE_NATIVE, P.LBM_USOLVE_F64) for g in (0.0, 0.2)]
    lines = ["%d %d %d %d %d %d %g" % ((lat,) + d + (st, pr, g)) for lat, dims, st, pr, g in sets for d in dims]
    keys = iter(_run(tmp_path, KEYS, "\n".join(lines)))
    seen = set()
    for lat, dims, st, pr, g in sets:
        got = [next(keys) for _ in dims]
        pairwise = lat == P.LBM_D3Q59 and st == P.LBM_STORE_F32_DEV and pr == P.LBM_USOLVE_NATIVE
        assert len(set(got)) == (3 if pairwise else 1), (lat, st, pr, g, got)
        if not (st == P.LBM_STORE_F64 and pr == P.LBM_USOLVE_F64):  # FP64 storage sweeps in FP64 either way
            assert not seen & set(got)
        seen |= set(got)
