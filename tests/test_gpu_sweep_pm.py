"""The u-solve sweep of the 3D FP32 deviations (pressure pair from the force kernel) against the FP64 run: copies
of one, two and four columns, tiles with and without tensor copies, lattices smaller than a tile's halo,
both equations of state."""
import numpy as np
import pytest

import paper_1402_2920_gb300 as P
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(case, eos, storage, rho, u, steps, **kw):
    prm = P.make_params(kappa=case.kappa, rho0=case.rho0, storage=storage, **kw)
    g = P.Sim(case.lattice, case.dims, eos, prm)
    g.init(rho, u)
    g.step(steps)
    st = g.stats()
    assert st.status == 0
    out = g.fields() + (st,)
    g.close()
    return out


# nx odd, 2 mod 4 and 0 mod 4; below a halo; several tiles with interior ones (nx >= 72, ny >= 24) and z slabs
@pytest.mark.parametrize("dims", [(4, 4, 4), (5, 7, 6), (33, 9, 5), (70, 24, 6), (72, 24, 37), (104, 33, 9)])
@pytest.mark.parametrize("kind", [P.LBM_EOS_VDW, P.LBM_EOS_PSI_SINE])
@pytest.mark.parametrize("solver", ["plain", "fast"])
def test_matches_fp64(dims, kind, solver):
    case = W.make_case("droplet3d", dims=dims)
    if kind == P.LBM_EOS_VDW:
        a, b, T = case.eos_abT
        eos = P.make_eos(kind, a=a, b=b, T=T)
    else:
        eos = P.make_eos(kind, rho1=0.5, rho2=1.0, A=0.4, cs2_rho1=0.5)
    y = np.arange(dims[1])[None, :, None]
    u = np.zeros((3,) + case.rho.shape) + np.array([0.01, -0.005, 0.012])[:, None, None, None]
    u[2] += 0.01 * np.sin(2 * np.pi * y / dims[1])
    kw = {"plain": {}, "fast": {"usolve_omega": 0.0, "usolve_chebyshev": 1, "usolve_warm_start": 2}}[solver]
    rho_d, u_d, _ = _run(case, eos, P.LBM_STORE_F64, case.rho, u, 3, **kw)
    rho_s, u_s, st = _run(case, eos, P.LBM_STORE_F32_DEV, case.rho, u, 3, **kw)
    interior = dims[0] % 4 == 0 and dims[0] >= 72 and dims[1] >= 24
    assert st.usolve_tensor_copies == (1 if interior else 0)
    # as for the pairwise kernels: rounding of the stored deviations and the solve's tolerance
    assert np.abs(rho_s - rho_d).max() < 2e-7
    assert np.abs(u_s - u_d).max() < 2e-7
