"""lbm_profile times the sweep that an accelerated solve runs: a Chebyshev sweep that reads the update before it; and a
plain one where the solve is plain."""
import re

import numpy as np
import pytest

import paper_1402_2920_gb300 as P
from gpu_util import lib_sim
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [P.LBM_STORE_F32_DEV, P.LBM_STORE_F16_LOC, P.LBM_STORE_F64])
@pytest.mark.parametrize("chebyshev", [0, 1])
def test_profiled_sweep_is_the_steps(storage, chebyshev, capfd, monkeypatch):
    case = W.make_case("droplet3d", dims=(24, 20, 16))
    monkeypatch.setenv("LBM_TRACE", "1")
    runs = []
    for profile in (False, True):
        g = lib_sim(case, storage=storage, warm=2, omega=0.0, chebyshev=chebyshev)
        g.init(case.rho)
        g.step(2)
        if profile:
            capfd.readouterr()
            ms = P.lbm_profile(g.handle, 3)
            assert all(v > 0 for v in ms.values())
            c1, c2 = (float(v) for v in re.search(r"lbm profile sweep c1 (\S+) c2 (\S+)", capfd.readouterr().err).groups())
            assert (c1 != 0.0) == bool(chebyshev) and c2 > 0.0
        g.step(2)
        runs.append(g.populations())
        g.close()
    assert np.array_equal(*runs)  # the profile left the state as it was
