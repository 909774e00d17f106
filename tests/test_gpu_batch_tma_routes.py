"""The ensemble's TMA mode with walls, outflow or a frozen temperature, and with columns of more than 60
planes (two halves): every instance has the state of its own context bit for bit, on the TMA kernel where
its columns fill the GPU and on the generic kernel where they do not."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

P, WALL, OUT, TH = W.BC_PERIODIC, W.BC_WALL, W.BC_OUTFLOW, W.BC_THERMAL_ONLY
# routes: items of a TMA column are whole or half columns, of the generic kernel 8 planes of 32 x 8 tiles
SMALL = [(24, 24, 24), (33, 9, 17), (5, 3, 2), (20, 21, 62)]
LARGE = [(33, 33, 64), (34, 33, 61), (33, 35, 63), (35, 33, 64)] * 3 + [(33, 33, 59), (5, 4, 3)]
CASES = {"periodic halves": ((P,) * 6, {}, [(40, 36, 70), (33, 24, 64), (24, 20, 61), (24, 20, 60)], True),
         "small box": ((WALL,) * 6, {}, SMALL, False), "box": ((WALL,) * 6, {}, LARGE, True),
         "walls x, open y": ((WALL, WALL, OUT, OUT, WALL, OUT), {}, LARGE, True),
         "box, 16 bits": ((WALL,) * 6, dict(precision=1, rho_ref=0.4, T_ref=0.0627), LARGE, True),
         "small frozen": ((P, P, P, P, WALL, OUT), dict(thermal_off=1), SMALL, False),
         "frozen": ((P, P, P, P, WALL, OUT), dict(thermal_off=1), LARGE, True),
         "frozen box": ((WALL,) * 6, dict(thermal_off=1), LARGE, True),
         "thermal faces": ((TH,) * 6, {}, SMALL, True)}


def _generic_items(dims):
    """items of the generic kernel: blocks of whole columns cut into chunks of at least 8 planes"""
    return sum(-(-x // 32) * -(-y // 8) * -(-z // 8) for x, y, z in dims)


@pytest.mark.parametrize("name", list(CASES))
def test_tma_mode_matches_single_contexts(name):
    from paper_2201_06039_gb300 import lbm
    bc, kw, dims, tma = CASES[name]
    setups = [W.LatticeSetup(*d, bc=bc, T_wall_over_Tc=(0.86, 0.87, 0.865, 0.855, 0.88, 0.86), sigma=W.SIGMA_STAR,
                             gravity=(1e-6, 0, -3e-5)) for d in dims]
    rng = np.random.default_rng(W.MASTER_SEED)
    Tc = lbm.lbm_eos_critical(lbm.params_from_setup(setups[0]))[0]
    rho = [(0.38 + 2e-3 * rng.random(s.shape)).astype(np.float32) for s in setups]
    T = [np.full(s.shape, 0.86 * Tc, np.float32) for s in setups]
    b = lbm.Batch(lbm.params_from_setup(setups[0], **kw), dims)
    b.select_plan(0, 0)
    assert (b.plan["items"] < _generic_items(dims) / 2) == tma, b.plan
    b.init(rho, T)
    b.step(1)
    b.step(11)     # a replayed chain of eight and three enqueued
    got = b.moments()
    sums = b.totals()
    b.select_plan(8, 1)
    b.step(2)      # into the persistent kernel and back
    b.select_plan(0, 0)
    b.step(9)
    later = b.moments()
    b.close()
    for k in {dims.index(d) for d in dims}:
        lat = lbm.Lattice(lbm.params_from_setup(setups[k], kernel=2, use_tma=0, **kw))
        lat.init(rho[k], T[k])
        for steps, have in ((12, got[k]), (11, later[k])):
            lat.step(steps)
            want = lat.moments()
            for f in want:
                assert np.isfinite(want[f]).all()
                assert np.array_equal(have[f], want[f]), (name, dims[k], steps, f)
        lat.close()
        assert np.isfinite(sums[k]).all()
