"""lbm_stats_get's sums against FP64 sums of the exported populations, for every storage and both lattices, at
site counts below, at and above one pass of the reduction's grid (1024 x 256 sites)."""
import numpy as np
import pytest

import paper_1402_2920_gb300 as P
from gpu_util import lib_sim
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STORAGES = [P.LBM_STORE_F32, P.LBM_STORE_F32_DEV, P.LBM_STORE_F16_DEV, P.LBM_STORE_BF16_DEV, P.LBM_STORE_F64,
            P.LBM_STORE_F32_LOC, P.LBM_STORE_F16_LOC, P.LBM_STORE_BF16_LOC]


@pytest.mark.parametrize("name,dims", [("droplet2d", (33, 17)), ("droplet2d", (512, 513)), ("droplet3d", (9, 7, 5)),
                                       ("droplet3d", (64, 64, 64)), ("droplet3d", (66, 65, 64))])
@pytest.mark.parametrize("storage", STORAGES)
def test_sums_match_the_populations(name, dims, storage):
    case = W.make_case(name, dims=dims)
    d = len(dims)
    u = np.zeros((d,) + case.rho.shape) + np.array([0.01, -0.02, 0.015])[:d].reshape((d,) + (1,) * d)
    g = lib_sim(case, storage=storage)
    g.init(case.rho, u)
    g.step(1)
    n = g.populations()
    st = g.stats()
    c = P.lbm_velocities(case.lattice)[:, :d]
    # both sides add the same stored values; what they leave is rounding, at most 2^-48 of the deviations
    # (and of n_i in the reference's FP64 sums) per site
    mass = n.sum()
    assert abs(st.mass - mass) < 1e-13 * mass
    for a in range(d):
        ref = (n.sum(axis=1) * c[:, a]).sum()
        assert abs(ref) > 1e-3 * mass
        assert abs(st.mom[a] - ref) < 1e-12 * mass
    g.close()
