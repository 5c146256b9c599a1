"""The 3D FP32-deviation kernels at a caller's own tolerances of the u-solve: the relative stop against the FP64 run with
the same stop, and loose absolute stops against the converged FP64 run."""
import numpy as np
import pytest

import paper_1402_2920_gb300 as P
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _case(dims):
    case = W.make_case("droplet3d", dims=dims)
    z = np.arange(dims[2])[:, None, None]
    u = np.zeros((3,) + case.rho.shape) + np.array([0.01, -0.012, 0.008])[:, None, None, None]
    u[0] += 0.02 * np.sin(2 * np.pi * z / dims[2])
    return case, u


def _run(case, storage, u, steps, **kw):
    a, b, T = case.eos_abT
    prm = P.make_params(kappa=case.kappa, rho0=case.rho0, storage=storage, **kw)
    g = P.Sim(case.lattice, case.dims, P.make_eos(P.LBM_EOS_VDW, a=a, b=b, T=T), prm)
    g.init(case.rho, u)
    g.step(steps)
    st = g.stats()
    assert st.status == 0
    out = g.fields()
    g.close()
    return out, st


@pytest.mark.parametrize("dims", [(5, 7, 6), (33, 9, 11), (75, 24, 9)])  # nx odd: the sweep alone differs in form
@pytest.mark.parametrize("rtol", [1e-2, 1e-4])
def test_relative_stop(dims, rtol):
    case, u = _case(dims)
    kw = {"usolve_rtol": rtol, "usolve_warm_start": 1}
    (rho_d, u_d), st_d = _run(case, P.LBM_STORE_F64, u, 3, **kw)
    (rho_s, u_s), st_s = _run(case, P.LBM_STORE_F32_DEV, u, 3, **kw)
    # the same sweeps, so the same iterates up to the rounding of the stored deviations, as for converged solves
    assert st_s.usolve_sweeps_total == st_d.usolve_sweeps_total
    assert 0.0 < st_s.usolve_resid < 1.0
    assert np.abs(rho_s - rho_d).max() < 2e-7
    assert np.abs(u_s - u_d).max() < 2e-7


@pytest.mark.parametrize("dims", [(34, 9, 11), (128, 24, 6)])  # pairwise kernels, 64-wide tiles; with tensor copies
@pytest.mark.parametrize("tol", [1e-6, 1e-5, 1e-4])
def test_loose_absolute_stop(dims, tol):
    case, u = _case(dims)
    (rho_d, u_d), _ = _run(case, P.LBM_STORE_F64, u, 3)
    (rho_s, u_s), st = _run(case, P.LBM_STORE_F32_DEV, u, 3, usolve_tol=tol, usolve_warm_start=1)
    assert st.usolve_resid <= tol
    # each of the three steps and the fields' own solve leave j~ within tol / (1 - 0.7) of the fixed point
    assert np.abs(rho_s - rho_d).max() < 2e-7 + 4 * tol / 0.3
    assert np.abs(u_s - u_d).max() < 2e-7 + 4 * tol / 0.3
