"""Populations in and out in FP64: the conversions give what FP64 arithmetic gives, also for zeros, subnormal
values, values that round up to the next power of two, and values beyond the float range."""
import numpy as np
import pytest

import paper_1402_2920_gb300 as P
from gpu_util import lib_sim
from paper_1402_2920_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,dims", [("droplet2d", (9, 7)), ("droplet3d", (6, 5, 4))])
def test_float_populations_round_to_nearest_even(name, dims):
    case = W.make_case(name, dims=dims)
    g = lib_sim(case, storage=P.LBM_STORE_F32)  # stored as float, no reference subtracted
    rng = np.random.default_rng(11)
    n = rng.standard_normal((g.Q, g.N)) * 10.0 ** rng.uniform(-44, 37, (g.Q, g.N))
    n[1, :8] = [0.0, -0.0, 1e-45, -1e-40, 1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24, 2.0 - 2.0 ** -30, 1.1754943e-38]
    n[2, :4] = [3.4028235e38, 3.4028236e38, -1e39, 2.0 ** -126 - 2.0 ** -160]
    with np.errstate(over="ignore"):
        ref = n.astype(np.float32).astype(np.float64)
    g.set_populations(n)
    out = g.populations()
    g.close()
    assert np.array_equal(out[1:], ref[1:])
    assert np.array_equal(np.signbit(out[1:]), np.signbit(ref[1:]))


@pytest.mark.parametrize("storage", [P.LBM_STORE_F32_DEV, P.LBM_STORE_F16_DEV, P.LBM_STORE_BF16_DEV,
                                     P.LBM_STORE_F32_LOC, P.LBM_STORE_F16_LOC, P.LBM_STORE_BF16_LOC, P.LBM_STORE_F64])
def test_transfer_is_idempotent(storage):
    """What comes out goes in again unchanged: each conversion is exact on values the storage holds."""
    case = W.make_case("droplet3d", dims=(10, 7, 6))
    g = lib_sim(case, storage=storage)
    g.init(case.rho)
    a = g.populations()
    g.set_populations(a)
    b = g.populations()
    g.close()
    tol = {P.LBM_STORE_F64: 0.0}.get(storage, 2.0 ** -50)  # the local reference is re-made from the sum
    if storage in (P.LBM_STORE_F32_LOC, P.LBM_STORE_F16_LOC, P.LBM_STORE_BF16_LOC):
        tol = {P.LBM_STORE_F32_LOC: 2.0 ** -23, P.LBM_STORE_F16_LOC: 2.0 ** -14, P.LBM_STORE_BF16_LOC: 2.0 ** -11}[storage]
    assert np.abs(a - b).max() <= tol
