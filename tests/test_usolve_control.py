"""The u-solve's control (csrc/lbm_usolve.h) on a model of the iteration, on the host.

The model keeps the residual of the linear iteration in the eigenvectors of its matrix J: a sweep adds
d = c1 d_prev + c2 r and leaves r - (1 - J) d of each mode.  A run is a series of solves whose first residuals
decline, as those of a settling flow do; Chebyshev sweeps throughout (cheb = 2) are what it is measured against."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MODEL = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "lbm_usolve.h"
using namespace lbm;

// argv: cheb maxit g smooth_share rough_share first_residual decline solves rounding
int main(int, char** a)
{
    const int cheb = std::atoi(a[1]), maxit = std::atoi(a[2]), solves = std::atoi(a[8]);
    const double g = std::atof(a[3]), smooth = std::atof(a[4]), rough = std::atof(a[5]), decline = std::atof(a[7]);
    const double rounding = std::atof(a[9]), lim = 5e-9;
    double first = std::atof(a[6]);
    constexpr int M = 64;  // modes 0 .. M/2: smooth, J of at most g/20; the others: up to g
    UsolveState u{};
    unsigned seed = 1;
    for (int s = 0; s < solves; ++s, first *= decline) {
        double J[M], r[M], d[M], total = 0.0;
        for (int k = 0; k < M; ++k) {
            const bool fine = k < M / 2;
            J[k] = g * (fine ? 0.05 * k / (M / 2) : double(k - M / 2 + 1) / (M / 2));
            r[k] = fine ? smooth : rough;
            d[k] = 0.0;
            total += r[k];
        }
        for (int k = 0; k < M; ++k) r[k] *= first / total;
        usolve_open(u, u, cheb, 0.0, maxit, g);
        const int opened = (u.opened & US_PLAIN) != 0;
        int missing = 0, unread = 0;  // sweeps that read an update none left; plain sweeps that leave theirs
        bool kept = false;
        while (u.iter < 1000) {
            double norm = 0.0;
            for (int k = 0; k < M; ++k) norm += std::fabs(r[k]);
            seed = seed * 1664525u + 1013904223u;
            norm += rounding * (seed >> 8) / 16777216.0;  // what the rounding of u puts into the residual
            missing += u.c1 != 0.0 && !kept;
            kept = keeps_update(u);
            unread += kept && u.mode != 1;
            for (int k = 0; k < M; ++k) {
                d[k] = u.c1 * d[k] + u.c2 * r[k];
                r[k] -= (1.0 - J[k]) * d[k];
            }
            u.iter += 1;
            const bool stop = norm <= lim;
            if (cheb && !stop) usolve_next(u, cheb, norm, lim);
            if (stop) usolve_end(u);
            u.resid_last = norm;
            u.resid_min = norm < u.resid_min ? norm : u.resid_min;
            if (stop) break;
        }
        u.iters_last = u.iter;
        std::printf("%d %d %d %d\n", opened, u.iter, missing, unread);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("usolve")
    src = d / "model.cpp"
    src.write_text(MODEL)
    exe = d / "model"
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1402_2920_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)

    def run(cheb, g, smooth, rough, first, decline, solves, rounding=0.0, maxit=500):
        out = subprocess.run([str(exe)] + [str(v) for v in (cheb, maxit, g, smooth, rough, first, decline, solves, rounding)],
                             check=True, capture_output=True, text=True).stdout
        rows = [[int(v) for v in line.split()] for line in out.splitlines()]
        assert not any(r[2] or r[3] for r in rows)  # the update vector: written before it is read, by no plain sweep
        return [r[1] for r in rows], [r[0] for r in rows]

    return run


@pytest.mark.parametrize("g", [0.4, 0.6, 0.8, 0.95])
@pytest.mark.parametrize("decline", [0.8, 0.9, 0.97, 1.0])
@pytest.mark.parametrize("first", [3e-4, 3e-6, 1e-7])
def test_noise_takes_no_more_sweeps_than_chebyshev(model, g, decline, first):
    """Noise on all modes alike: plain sweeps gain nothing, and looking for it costs one sweep of a solve at
    most, and over a run of 60 solves no more than one in twenty."""
    ref, _ = model(2, g, 1.0, 1.0, first, decline, 60)
    got, _ = model(1, g, 1.0, 1.0, first, decline, 60)
    assert max(b - a for a, b in zip(ref, got)) <= 1
    assert sum(got) <= 1.05 * sum(ref) + 1


@pytest.mark.parametrize("g", [0.4, 0.6, 0.8])
@pytest.mark.parametrize("first", [2e-8, 2e-7, 1e-6])
def test_smooth_flow_goes_over_to_plain_sweeps(model, g, first):
    """A steady smooth residual with a thousandth of noise: within a few solves the sweeps are plain, and
    take no more than the plain iteration needs."""
    ref, _ = model(2, g, 1.0, 1e-3, first, 1.0, 40)
    plain, _ = model(0, g, 1.0, 1e-3, first, 1.0, 40)
    got, opened = model(1, g, 1.0, 1e-3, first, 1.0, 40)
    assert max(got) <= max(ref) + 1
    if ref[-1] <= 5:
        assert opened[-1] and got[-1] <= min(ref[-1], plain[-1])


@pytest.mark.parametrize("g", [0.5, 0.6, 0.9])
def test_rounding_of_u_does_not_stall_a_solve(model, g):
    """Residuals that rounding keeps between a half of the tolerance and just above it."""
    for smooth, rough in ((1.0, 1e-3), (1.0, 1.0)):
        got, _ = model(1, g, smooth, rough, 1e-7, 1.0, 200, rounding=4.5e-9)
        assert max(got) <= 16


@pytest.mark.parametrize("maxit", [3, 5, 10])
def test_a_tight_cap_keeps_chebyshev(model, maxit):
    """A solve that Chebyshev ends within the caller's cap is not opened with a sweep that could exceed it."""
    _, opened = model(1, 0.6, 1.0, 1e-3, 2e-7, 1.0, 40, maxit=maxit)
    assert not any(opened)
