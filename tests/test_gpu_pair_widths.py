"""The pairwise kernels at the widths that their tile rule chooses: 64-wide tiles with a last tile of one pair, and
lattices of one tile, against the FP64 run."""
import numpy as np
import pytest

import paper_1402_2920_gb300 as P
from paper_1402_2920_gb300 import workloads as W
from test_gpu_pair_kernels import _eos, _run

pytestmark = pytest.mark.gpu


# 130: two 64-wide tiles and one pair; 34, 62: one 64-wide tile; 98: two; 66: two 32-wide tiles and one pair
@pytest.mark.parametrize("dims", [(130, 5, 6), (34, 5, 7), (62, 4, 5), (66, 9, 4), (98, 7, 5)])
@pytest.mark.parametrize("gamma", [0.0, 0.2])
def test_pairs_match_fp64(dims, gamma):
    case = W.make_case("droplet3d", dims=dims)
    rng = np.random.default_rng(6)
    y = np.arange(dims[1])[None, :, None]
    u = np.zeros((3,) + case.rho.shape) + np.array([-0.01, 0.007, 0.011])[:, None, None, None]
    u[2] += 0.01 * np.sin(2 * np.pi * y / dims[1])
    rho = case.rho + 1e-4 * rng.uniform(-1, 1, case.rho.shape)
    eos = _eos(P.LBM_EOS_VDW, case)
    for d, s in zip(_run(case, eos, P.LBM_STORE_F64, gamma, rho, u, 4), _run(case, eos, P.LBM_STORE_F32_DEV, gamma, rho, u, 4)):
        assert np.abs(s - d).max() < 2e-7  # as the tests of the kernels' other sizes
