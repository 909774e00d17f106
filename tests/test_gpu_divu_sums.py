"""The rho_ave of a step with finite-difference div u is an FP64 sum from the node on, and the step is
the same for every size of lattice."""
import math

import numpy as np
import pytest

import workloads as W
from tests._parity import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("thermal_q", [7, 19])
def test_rho_ave_of_a_finite_difference_step_is_an_fp64_sum(thermal_q):
    """A step sums the rho of the state it starts from (the bits lbm_get_moments gives for it).  Bound of an
    FP64 sum of positive terms: at most 64 additions deep (16 planes a thread, 5 + 8 in a block, up to 23
    partials a thread, 5 + 8 again), each rounding by 2^-53 of the sum; the exact sum by math.fsum."""
    from paper_2201_06039_gb300 import lbm
    # a drop in vapour: sums of a column that go from vapour to liquid lose bits in 32-bit pairs
    s = W.LatticeSetup(96, 96, 64, sigma=W.SIGMA_STAR, gravity=(0.0, 0.0, -1e-6), divu_mode=1)
    case = dict(name="drop", setup=s, kind="droplet", R0=22.0, W=4.0, Tr_drop=0.86, Tr_gas=0.86, noise=1e-3,
                noise_seed=W.MASTER_SEED + 3)
    rho, T, _ = inputs(case)
    lat = lbm.Lattice(lbm.params_from_setup(s, thermal_q=thermal_q))
    lat.init(rho.astype(np.float32), T.astype(np.float32))
    lat.step(3)
    exact = math.fsum(lat.moments()["rho"].ravel().tolist()) / lat.N
    lat.step(1)
    rho_ave = lat.totals()[2]
    lat.close()
    assert abs(rho_ave - exact) <= 64 * 2.0 ** -53 * exact, (rho_ave, exact, rho_ave / exact - 1)
