"""The derivative and collision kernels on pairs of sites (3D, FP32 deviations, nx even) against the same
run in FP64, at the edges of their tiles (32 x 8 and 64 x 4 sites) and for both equations of state, and their
independence of which word of a pair a site is."""
import numpy as np
import pytest

import paper_1402_2920_gb300 as P
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(case, eos, storage, gamma, rho, u, steps):
    prm = P.make_params(gamma=gamma, kappa=case.kappa, rho0=case.rho0, storage=storage, usolve_omega=0.0,
                        usolve_chebyshev=1, usolve_warm_start=2)
    g = P.Sim(case.lattice, case.dims, eos, prm)
    g.init(rho, u)
    g.step(steps)
    assert g.stats().status == 0
    out = g.fields() + (g.populations(),)
    g.close()
    return out


def _eos(kind, case):
    if kind == P.LBM_EOS_VDW:
        a, b, T = case.eos_abT
        return P.make_eos(kind, a=a, b=b, T=T)
    # a stiffening psi-sine fluid whose interval holds the whole density range of the droplet
    return P.make_eos(kind, rho1=0.5, rho2=1.0, A=0.4, cs2_rho1=0.5)


# one tile in part (4), one more pair than a tile (34, 66), tiles exactly (64, 128), a padded last tile (96: 32 wide;
# 90: 64 wide; 160: 64 wide); y and z ragged against 4, 8 and the slab depth
@pytest.mark.parametrize("dims", [(4, 4, 4), (6, 5, 9), (34, 9, 7), (62, 7, 12), (64, 8, 33), (66, 13, 5), (90, 6, 6),
                                  (96, 11, 4), (128, 5, 10), (160, 4, 5)])
@pytest.mark.parametrize("kind,gamma", [(P.LBM_EOS_VDW, 0.0), (P.LBM_EOS_VDW, 0.2), (P.LBM_EOS_PSI_SINE, 0.0)])
def test_pairs_match_fp64(dims, kind, gamma):
    case = W.make_case("droplet3d", dims=dims)
    rng = np.random.default_rng(5)
    z = np.arange(dims[2])[:, None, None]
    u = np.zeros((3,) + case.rho.shape) + np.array([0.01, -0.012, 0.008])[:, None, None, None]
    u[0] += 0.01 * np.sin(2 * np.pi * z / dims[2])
    rho = case.rho + 1e-4 * rng.uniform(-1, 1, case.rho.shape)
    eos = _eos(kind, case)
    rho_d, u_d, n_d = _run(case, eos, P.LBM_STORE_F64, gamma, rho, u, 4)
    rho_s, u_s, n_s = _run(case, eos, P.LBM_STORE_F32_DEV, gamma, rho, u, 4)
    # rho is handed out as the float rho0 + drho (6e-8) and moves by the rounding of the stored deviations,
    # 2^-24 sum_i |dev_i| (about 1e-8 a step); u moves by that and by the solve's 5e-9 / (1 - 0.7) a step
    assert np.abs(rho_s - rho_d).max() < 2e-7
    assert np.abs(u_s - u_d).max() < 2e-7
    assert np.abs(n_s - n_d).max() < 2e-7


@pytest.mark.parametrize("gamma", [0.0, 0.15])
@pytest.mark.parametrize("dims", [(34, 6, 5), (66, 5, 6)])
def test_odd_shifts_move_the_bits(dims, gamma):
    case = W.make_case("spinodal3d", dims=dims)
    a, b, T = case.eos_abT
    eos = P.make_eos(P.LBM_EOS_VDW, a=a, b=b, T=T)
    ref = _run(case, eos, P.LBM_STORE_F32_DEV, gamma, case.rho, None, 3)
    for sh in ((0, 0, 1), (2, 1, 3)):
        got = _run(case, eos, P.LBM_STORE_F32_DEV, gamma, np.ascontiguousarray(np.roll(case.rho, sh, axis=(0, 1, 2))),
                   None, 3)
        assert np.array_equal(np.roll(ref[0], sh, axis=(0, 1, 2)), got[0])
        n = ref[2].reshape((59,) + case.rho.shape)
        assert np.array_equal(np.roll(n, sh, axis=(1, 2, 3)).reshape(59, -1), got[2])
