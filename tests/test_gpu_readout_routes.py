"""lbm_get_moments takes one of three routes (the TMA kernel's read-out, k_readout, a psi and a moments pass)
by size, faces and state: all give the same bits.  Sizes lie on both sides of each line, with no
extent a multiple of a tile."""
import numpy as np
import pytest

import workloads as W
from tests._parity import inputs

pytestmark = pytest.mark.gpu

P, WALL, OUT, TH = W.BC_PERIODIC, W.BC_WALL, W.BC_OUTFLOW, W.BC_THERMAL_ONLY
FACES = {"periodic": (P,) * 6, "pool": (P, P, P, P, WALL, OUT), "box": (WALL,) * 6, "corners": (WALL, OUT, OUT, WALL, WALL, OUT),
         "thermal x": (TH, TH, P, P, TH, TH), "open y": (P, P, OUT, OUT, WALL, WALL)}


def _state(dims, faces, **kw):
    nx, ny, nz = dims
    s = W.LatticeSetup(nx, ny, nz, bc=FACES[faces], T_wall_over_Tc=(0.86, 0.87, 0.865, 0.855, 0.88, 0.86), sigma=W.SIGMA_STAR,
                       gravity=(1e-6, 2e-6, -3e-5), hot_dT_over_Tc=0.05, hot_sigma=4.0, **kw)
    rho, T, _ = inputs(dict(name="read-out", setup=s, kind="pool", height=nz / 2.0, W=4.0, Tr_liquid=0.86, noise=1e-3,
                            noise_seed=W.MASTER_SEED + nx))
    return s, rho.astype(np.float32), T.astype(np.float32)


def _same(got, want, what):
    for k in want:
        assert np.isfinite(want[k]).all()
        assert np.array_equal(got[k], want[k]), (what, k)


BITS16 = dict(rho_ref=3.0, T_ref=0.06)
WET = dict(wall_scheme=1, wall_phi=1.1, wall_drho=0.05)


@pytest.mark.parametrize("faces,kw,wet", [("periodic", {}, False), ("pool", {}, False), ("box", {}, False), ("corners", {}, False),
                                          ("thermal x", {}, False), ("open y", {}, False), ("pool", {}, True), ("box", {}, True),
                                          ("pool", dict(precision=1, **BITS16), False), ("box", dict(precision=1, **BITS16), False),
                                          ("corners", dict(precision=2, **BITS16), False),
                                          ("periodic", dict(precision=2, **BITS16), False),
                                          ("pool", dict(thermal_off=1), True)])
@pytest.mark.parametrize("dims", [(67, 53, 41), (80, 50, 36)])
def test_tma_readout_is_that_of_the_generic_kernel(dims, faces, kw, wet):
    from paper_2201_06039_gb300 import lbm
    assert np.prod(dims) >= 1 << 17
    s, rho, T = _state(dims, faces, **(WET if wet else {}))
    tma = lbm.Lattice(lbm.params_from_setup(s, kernel=2, use_tma=1, **kw))
    gen = lbm.Lattice(lbm.params_from_setup(s, kernel=2, use_tma=0, **kw))
    assert (tma.kernel, gen.kernel) == (lbm.LBM_KERNEL_FUSED_TMA, lbm.LBM_KERNEL_FUSED)
    tma.init(rho, T)
    shapes = lbm.lbm_plan_shapes()
    # the model's plan, the read-out's own tile shape as the step's, and another one: its maps stay right
    for steps, shape in ((0, None), (4, None), (3, shapes.index((32, 12))), (3, shapes.index((24, 16)))):
        if shape is not None:
            tma.select_plan(shape, 5)
        tma.step(steps)
        gen.load_state(tma.save_state())
        _same(tma.moments(), gen.moments(), (steps, shape))
    tma.close()
    gen.close()


# (route by size; z extents 1 to 4 and 8 and 9 around the thin lattices' lines)
THIN = [(260, 256, 1), (259, 256, 1), (300, 220, 2), (161, 137, 3), (150, 110, 3), (201, 171, 4), (150, 119, 8), (129, 117, 9)]


@pytest.mark.parametrize("faces,kw", [("periodic", {}), ("box", {}), ("corners", {}), ("pool", dict(thermal_off=1)),
                                      ("box", dict(precision=1, **BITS16)), ("periodic", dict(precision=2, **BITS16))])
@pytest.mark.parametrize("dims", THIN)
def test_thin_readout_is_that_of_the_ensemble(dims, faces, kw):
    """The ensemble reads out through k_readout whatever the size."""
    from paper_2201_06039_gb300 import lbm
    if dims[2] == 1 and OUT in FACES[faces][4:]:
        pytest.skip("an outflow face needs two nodes across")
    s, rho, T = _state(dims, faces)
    lat = lbm.Lattice(lbm.params_from_setup(s, **kw))
    b = lbm.Batch(lbm.params_from_setup(s, **kw), [dims])
    lat.init(rho, T)
    b.init([rho], [T])
    for steps in (0, 3):
        lat.step(steps)
        b.step(steps)
        _same(lat.moments(), b.moments()[0], steps)
    lat.close()
    b.close()


@pytest.mark.parametrize("nz", [1, 2, 3])
def test_thin_readout_on_the_d3q19_temperature_lattice(nz):
    """A z-periodic slab of nz planes is four of them on top of each other (read out by k_readout)."""
    from paper_2201_06039_gb300 import lbm
    s, rho, T = _state((299, 221, nz), "periodic")
    s4, _, _ = _state((299, 221, 4 * nz), "periodic")
    # (a fixed rho_b: the domain means of the two round differently)
    one, four = (lbm.Lattice(lbm.params_from_setup(x, thermal_q=19, rho_buoy=0.4)) for x in (s, s4))
    one.init(rho, T)
    four.init(np.concatenate([rho] * 4), np.concatenate([T] * 4))
    for steps in (0, 3):
        one.step(steps)
        four.step(steps)
        a, b = one.moments(), four.moments()
        _same(a, {k: v[:nz] for k, v in b.items()}, steps)
    one.close()
    four.close()
