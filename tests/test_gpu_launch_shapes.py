"""The launch shapes that lbm_create chooses from the lattice give the same results as any other."""
import os

import numpy as np
import pytest

import paper_1402_2920_gb300 as P
from gpu_util import lib_sim
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(dims, storage, env, steps=3):
    old = {k: os.environ.get(k) for k in env}
    os.environ.update(env)
    try:
        case = W.make_case("droplet3d", dims=dims)
        rng = np.random.default_rng(7)
        u = 0.01 * rng.standard_normal((3,) + case.rho.shape)
        g = lib_sim(case, storage=storage, warm=2, omega=0.0, chebyshev=1)
        g.init(case.rho, u)
        g.step(steps)
        pops = g.populations()
        rho, v = g.fields()
        g.close()
        return pops, rho, v
    finally:
        for k, x in old.items():
            if x is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = x


# one plane per slab, slabs that divide the depth, a ragged last slab, one slab; a lattice thinner
# than a tile's halo and one with several tiles per row
@pytest.mark.parametrize("dims", [(4, 5, 4), (37, 19, 11), (68, 24, 9)])
@pytest.mark.parametrize("storage", [P.LBM_STORE_F32_DEV, P.LBM_STORE_F64])
def test_any_slab_depth_gives_the_chosen_depths_bits(dims, storage):
    ref = _run(dims, storage, {})
    for zb in (1, 2, dims[2] - 1, dims[2]):
        got = _run(dims, storage, {"LBM_TILE_Z": str(zb)})
        for a, b in zip(ref, got):
            assert np.array_equal(a, b)
