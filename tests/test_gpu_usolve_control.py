"""The accelerated u-solve's choice between Chebyshev and plain sweeps: same fixed point, within the
tolerance, for noise (Chebyshev from the start), for smooth flow (plain from the start) and for the
16-bit storages' tolerance, and no more sweeps than the plain iteration by more than its one opening."""
import numpy as np
import pytest

import paper_1402_2920_gb300 as P
from gpu_util import lib_sim, oracle_sim
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _flow(case, amplitude, noise):
    rng = np.random.default_rng(3)
    d = len(case.dims)
    u = noise * rng.standard_normal((d,) + case.rho.shape)
    y = np.arange(case.dims[1])
    u[0] += amplitude * np.sin(2 * np.pi * y / case.dims[1]).reshape((1,) * (d - 2) + (-1, 1))
    return u


@pytest.mark.parametrize("name,dims", [("droplet2d", (40, 33)), ("droplet3d", (18, 17, 12))])
@pytest.mark.parametrize("amplitude,noise", [(0.02, 0.0), (0.0, 0.005)])
@pytest.mark.parametrize("warm", [0, 1, 2])
def test_fixed_point_and_sweeps(name, dims, amplitude, noise, warm):
    case = W.make_case(name, dims=dims)
    u = _flow(case, amplitude, noise)
    o = oracle_sim(case)
    o.init(case.rho, u)
    assert o.step(6) == 0
    rho_o, u_o, _ = o.fields()
    sweeps = {}
    for cheb in (0, 1):
        g = lib_sim(case, storage=P.LBM_STORE_F64, warm=warm, omega=0.0 if cheb else 1.0, chebyshev=cheb)
        g.init(case.rho, u)
        g.step(6)
        st = g.stats()
        assert st.status == 0
        sweeps[cheb] = st.usolve_sweeps_total
        rho_g, u_g = g.fields()
        # each solve stops at |j~new - j~| <= 1e-14: its iterate is within 1e-14/(1 - 0.7) of the fixed
        # point, and six steps of a stable update keep the sum of such errors below 1e-12
        assert np.abs(rho_g - rho_o).max() < 1e-12
        assert np.abs(u_g - u_o[: u_g.shape[0]].reshape(u_g.shape)).max() < 1e-12
        g.close()
    assert sweeps[1] <= sweeps[0] + 6


@pytest.mark.parametrize("storage", [P.LBM_STORE_F32_DEV, P.LBM_STORE_F16_LOC])
def test_flow_at_the_rounding_of_u_still_converges(storage):
    """|u| of 0.04 rounds at 2e-9 in FP32, two fifths of the FP32 tolerance of 5e-9."""
    case = W.make_case("droplet3d", dims=(24, 20, 16))
    u = _flow(case, 0.04, 0.0)
    g = lib_sim(case, storage=storage, warm=2, omega=0.0, chebyshev=1)
    g.init(case.rho, u)
    g.step(12)
    st = g.stats()
    assert st.status == 0 and st.usolve_iters_max < 40
