"""Step graphs that a context keeps over lbm_init_fields and lbm_load_state: a replay must be one that
was captured for a state of the same form.  A frozen field stays as it was given, un-streamed after
lbm_init_fields and streamed after a checkpoint of a run in which it evolved, so the same (n, buffer,
sum slot) can come up with either form in one context."""
import numpy as np
import pytest

import workloads as W
from tests._parity import inputs

pytestmark = pytest.mark.gpu

P, WALL = W.BC_PERIODIC, W.BC_WALL


def _case():
    s = W.LatticeSetup(40, 24, 16, bc=(P, P, P, P, WALL, WALL), T_wall_over_Tc=(0.86,) * 4 + (0.88, 0.86),
                       sigma=W.SIGMA_STAR, gravity=(1e-6, 0, -3e-5), hot_dT_over_Tc=0.05, hot_sigma=4.0)
    rho, T, _ = inputs(dict(name="kept", setup=s, kind="pool", height=8.0, W=4.0, Tr_liquid=0.86, noise=1e-3,
                            noise_seed=W.MASTER_SEED + 5))
    return s, rho.astype(np.float32), T.astype(np.float32)


def _lattice(s, **kw):
    from paper_2201_06039_gb300 import lbm
    return lbm.Lattice(lbm.params_from_setup(s, kernel=kw.pop("kernel", 2), **kw))


def _expect(s, frozen, start, steps, kernel):
    """fields after `steps` steps of a context of its own, without graphs"""
    lat = _lattice(s, use_graph=0, kernel=kernel, **frozen)
    start(lat)
    lat.step(steps)
    m = lat.moments()
    lat.close()
    return m


@pytest.mark.parametrize("kernel", [1, 2])
@pytest.mark.parametrize("load_first", [True, False])
@pytest.mark.parametrize("frozen", ["thermal_off", "flow_off"])
def test_graphs_kept_over_init_and_load_match_the_state(frozen, load_first, kernel):
    s, rho, T = _case()
    src = _lattice(s, kernel=kernel)
    src.init(rho, T)
    src.step(4)
    ckpt = src.save_state()
    src.close()
    off = {frozen: 1}

    def load(lat):
        lat.load_state(ckpt)

    def init(lat):
        lat.init(rho, T)
    order = [load, init, load, init] if load_first else [init, load, init, load]
    lat = _lattice(s, use_graph=1, kernel=kernel, **off)
    for k, start in enumerate(order):
        start(lat)
        if start is load:   # from init the first of six steps is enqueued directly, the rest replayed
            lat.step(1)
            lat.step(5)
        else:
            lat.step(6)
        got = lat.moments()
        want = _expect(s, off, start, 6, kernel)
        for f in got:
            assert np.array_equal(got[f], want[f]), (k, start.__name__, f)
    lat.close()


def test_a_graph_kept_over_init_is_replayed():
    """An evolving context that runs one set of fields after another replays its graph: same results
    as a context of its own for each."""
    s, rho, T = _case()
    lat = _lattice(s, use_graph=1)
    for k in range(3):
        r = (rho * np.float32(1 + 1e-3 * k)).astype(np.float32)
        lat.init(r, T)
        lat.step(9)
        got = lat.moments()
        want = _expect(s, {}, lambda x: x.init(r, T), 9, 2)
        for f in got:
            assert np.array_equal(got[f], want[f]), (k, f)
    lat.close()
