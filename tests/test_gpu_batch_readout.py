"""The one-launch read-out of an ensemble against the read-out of each instance's own context, bit for bit,
for ensembles small enough to be cut into single planes and large enough for the longest chunks."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

P, WALL, OUT = W.BC_PERIODIC, W.BC_WALL, W.BC_OUTFLOW
# read-out chunks of 1, 2, 7 and 16 planes on 152 SMs
ENSEMBLES = {"one cube": [(32, 32, 32)], "a few": [(33, 17, 20), (24, 24, 24), (5, 3, 2), (20, 9, 41), (40, 20, 30)],
             "tall": [(40, 41, 70), (41, 33, 61)], "many": [(48, 40, 33)] * 6 + [(33, 50, 70)] * 5 + [(7, 9, 3)] * 3}


@pytest.mark.parametrize("faces", ["periodic", "box"])
@pytest.mark.parametrize("name", list(ENSEMBLES))
def test_readout_matches_single_contexts(name, faces):
    from paper_2201_06039_gb300 import lbm
    dims = ENSEMBLES[name]
    bc = (P,) * 6 if faces == "periodic" else (WALL, WALL, WALL, WALL, WALL, OUT)
    setups = [W.LatticeSetup(*d, bc=bc, T_wall_over_Tc=(0.86,) * 6, sigma=W.SIGMA_STAR, gravity=(1e-6, 0, -3e-5)) for d in dims]
    rng = np.random.default_rng(W.MASTER_SEED)
    Tc = lbm.lbm_eos_critical(lbm.params_from_setup(setups[0]))[0]
    rho = [(0.38 + 2e-3 * rng.random(s.shape)).astype(np.float32) for s in setups]
    T = [np.full(s.shape, 0.86 * Tc, np.float32) for s in setups]
    b = lbm.Batch(lbm.params_from_setup(setups[0]), dims)
    b.init(rho, T)
    for steps in (0, 3):      # un-streamed populations, then pulled ones
        b.step(steps)
        got = b.moments()
        for k in {dims.index(d) for d in dims}:
            lat = lbm.Lattice(lbm.params_from_setup(setups[k], kernel=2, use_tma=0))
            lat.init(rho[k], T[k])
            lat.step(steps)
            want = lat.moments()
            lat.close()
            for f in want:
                assert np.array_equal(got[k][f], want[f]), (name, dims[k], steps, f)
    b.close()
