"""Sweeps of the accelerated u-solve on the 3D spinodal of the benchmark's recipe: where the flow is noise, no more
than Chebyshev sweeps throughout take, and where it has become smooth, the plain sweeps' two."""
import pytest

import paper_1402_2920_gb300 as P
from gpu_util import lib_sim
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_sweeps_over_the_transient():
    case = W.make_case("spinodal3d", dims=(64, 64, 64))
    g = lib_sim(case, storage=P.LBM_STORE_F32_DEV, warm=2, omega=0.0, chebyshev=1)
    g.init(case.rho)
    total = []
    for n in (5, 20, 15, 8):
        g.step(n)
        st = g.stats()
        assert st.status == 0
        total.append(st.usolve_sweeps_total)
    g.close()
    # Chebyshev throughout: 117 sweeps over steps 6 to 25 on this lattice
    assert total[1] - total[0] <= 117
    assert total[3] - total[2] <= 16
