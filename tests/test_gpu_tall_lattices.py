"""A lattice with more rows than a grid of four-row tiles has CTAs (3D, FP32 deviations, nx even): it steps, and as a
periodic repetition of a small lattice it has the small lattice's fields, bit for bit."""
import pytest
import torch

import paper_1402_2920_gb300 as P
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _fields(case, eos, dims, rho, steps):
    prm = P.make_params(kappa=case.kappa, rho0=case.rho0, storage=P.LBM_STORE_F32_DEV, usolve_omega=0.0,
                        usolve_chebyshev=1, usolve_warm_start=2)
    g = P.Sim(case.lattice, dims, eos, prm, torch.cuda.current_stream().cuda_stream)
    g.init(rho)
    g.step(steps)
    out, u = torch.empty_like(rho), torch.empty((3,) + tuple(rho.shape), dtype=torch.float64, device="cuda")
    P.lbm_fields(g.handle, out, u, g.N, g.d)
    assert g.stats().status == 0
    g.close()
    return out, u


def test_repetition_in_y_has_the_small_lattices_fields():
    small, copies = (34, 32, 4), 8192
    case = W.make_case("spinodal3d", dims=small)
    a, b, T = case.eos_abT
    eos = P.make_eos(P.LBM_EOS_VDW, a=a, b=b, T=T)
    rho = torch.as_tensor(case.rho).cuda()
    ref, uref = _fields(case, eos, small, rho, 2)
    big, ubig = _fields(case, eos, (34, 32 * copies, 4), rho.repeat(1, copies, 1), 2)
    assert torch.equal(big.view(4, copies, 32, 34), ref[:, None].expand(-1, copies, -1, -1))
    assert torch.equal(ubig.view(3, 4, copies, 32, 34), uref[:, :, None].expand(-1, -1, copies, -1, -1))
