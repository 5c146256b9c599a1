"""lbm_profile leaves nothing behind that lbm_fields depends on: the fields after it are the same bits as without it."""
import numpy as np
import pytest

import paper_1402_2920_gb300 as P
from gpu_util import lib_sim
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [P.LBM_STORE_F32_DEV, P.LBM_STORE_F64])
@pytest.mark.parametrize("name,dims", [("spinodal3d", (24, 20, 16)), ("droplet2d", (40, 33))])
def test_fields_after_a_profile(name, dims, storage):
    case = W.make_case(name, dims=dims)
    runs = []
    for profile in (False, True):
        g = lib_sim(case, storage=storage, warm=2, omega=0.0, chebyshev=1)
        g.init(case.rho)
        g.step(1)
        if profile:
            P.lbm_profile(g.handle, 2)
        g.step(40)
        runs.append(g.fields())
        g.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
