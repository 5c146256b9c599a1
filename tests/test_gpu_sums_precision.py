"""The conservation sums keep FP64's precision and range in the storages that hold floats: one site's populations against
their exact sum, and values whose float sum overflows."""
import math

import numpy as np
import pytest

import paper_1402_2920_gb300 as P
from gpu_util import lib_sim
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [("droplet2d", (5, 4)), ("droplet3d", (5, 4, 4))]


def _sim(name, dims, storage=P.LBM_STORE_F32):
    case = W.make_case(name, dims=dims)
    return lib_sim(case, storage=storage), P.lbm_velocities(case.lattice)[:, :len(dims)].astype(np.float64)


@pytest.mark.parametrize("name,dims", CASES)
def test_one_sites_sums_are_exact_to_fp64_rounding(name, dims):
    g, c = _sim(name, dims)  # n_i itself as float
    rng = np.random.default_rng(2)
    for k in range(24):
        n = np.zeros((g.Q, g.N))
        n[:, (7 * k) % g.N] = rng.uniform(0.2, 1.0, g.Q) * 10.0 ** rng.uniform(-3, 0, g.Q)
        g.set_populations(n)
        out = g.populations()  # the floats that are stored
        st = g.stats()
        # the sum is taken in more than FP64's bits and converted: one rounding of its high part and one of the total
        mass = math.fsum(out.ravel())
        assert abs(st.mass - mass) <= 2.0 ** -52 * mass
        for a in range(c.shape[1]):
            t = (out * c[:, a:a + 1]).ravel()
            assert abs(st.mom[a] - math.fsum(t)) <= 2.0 ** -52 * math.fsum(np.abs(t))
    g.close()


@pytest.mark.parametrize("name,dims", CASES)
def test_range_beyond_float_sums(name, dims):
    g, c = _sim(name, dims)
    n = np.ones((g.Q, g.N))
    n[:, 3] = 3.0e38  # each a float, their sum none
    g.set_populations(n)
    out, st = g.populations(), g.stats()
    assert st.mass == pytest.approx(math.fsum(out.ravel()), rel=1e-14)
    for a in range(c.shape[1]):
        assert abs(st.mom[a]) <= 1e-14 * st.mass  # opposite velocities cancel
    n[2, 5] = np.inf
    g.set_populations(n)
    assert g.stats().mass == np.inf
    g.close()


@pytest.mark.parametrize("storage", [P.LBM_STORE_F32, P.LBM_STORE_F32_DEV, P.LBM_STORE_F32_LOC, P.LBM_STORE_F16_LOC])
def test_sums_over_many_sites_per_thread(storage):
    """Two sites to a thread: the total is that of the exported populations."""
    case = W.make_case("droplet3d", dims=(128, 64, 64))
    g = lib_sim(case, storage=storage)
    g.init(case.rho, np.zeros((3,) + case.rho.shape) + np.array([0.01, -0.02, 0.015])[:, None, None, None])
    g.step(1)
    n, st = g.populations(), g.stats()
    g.close()
    c = P.lbm_velocities(case.lattice).astype(np.float64)
    per = n.sum(axis=1, dtype=np.longdouble)
    # roundings: one of each exported population, two where a thread's sum is made a double, 8 levels of the
    # block's tree, 4 partial sums per thread of the last block and its 8 levels; four for the weights in the exports
    tol = 27 * 2.0 ** -53
    mass = per.sum()
    assert abs(st.mass - mass) <= tol * mass
    for a in range(3):
        assert abs(st.mom[a] - (per * c[:, a]).sum()) <= tol * (per * np.abs(c[:, a])).sum()
