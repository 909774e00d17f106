"""Ghost cells are refreshed by a kernel of their own only where the next launch reads them: not after
lbm_init_fields, not on lattices that wrap across neither x nor y, not behind the generic kernel on a
frozen temperature in streamed form.  The cells that are left alone hold NaN here."""
import numpy as np
import pytest

import workloads as W
from tests._parity import inputs

pytestmark = pytest.mark.gpu

P, WALL, OUT = W.BC_PERIODIC, W.BC_WALL, W.BC_OUTFLOW


def _setup(dims, bc, **kw):
    nx, ny, nz = dims
    s = W.LatticeSetup(nx, ny, nz, bc=bc, T_wall_over_Tc=(0.86, 0.87, 0.865, 0.855, 0.88, 0.86), sigma=W.SIGMA_STAR,
                       gravity=(1e-6, 0, -3e-5), hot_dT_over_Tc=0.05, hot_sigma=4.0, **kw)
    rho, T, _ = inputs(dict(name="ghosts", setup=s, kind="pool", height=nz / 2.0, W=4.0, Tr_liquid=0.86, noise=1e-3,
                            noise_seed=W.MASTER_SEED + nx))
    return s, rho.astype(np.float32), T.astype(np.float32)


def _lattice(s, **kw):
    import torch
    from paper_2201_06039_gb300 import lbm
    p = lbm.params_from_setup(s, kernel=2, **kw)
    poison = torch.full((lbm.lbm_workspace_bytes(p) + 256,), 255, dtype=torch.uint8, device="cuda")
    del poison   # the workspace takes this block: every float in it starts as a NaN
    return lbm.Lattice(p)


# dims, faces, options, refreshes expected of the first step and of the three after it
CASES = {"periodic, ghosts by TMA": ((64, 48, 6), (P,) * 6, {}, 1, 0),
         "periodic, ghosts stored directly": ((37, 11, 9), (P,) * 6, {}, 1, 0),
         "periodic, refreshed every step": ((20, 12, 9), (P,) * 6, dict(precision=1, rho_ref=3.0, T_ref=0.06), 1, 3),
         "walls across x": ((41, 19, 8), (WALL, WALL, P, P, WALL, OUT), {}, 1, 0),
         "walls across x and y": ((41, 19, 8), (WALL, WALL, WALL, WALL, P, P), {}, 0, 0),
         "open across x, walls across y": ((40, 24, 8), (OUT, OUT, WALL, WALL, WALL, OUT), {}, 0, 0),
         "closed, 16 bits": ((20, 12, 9), (WALL,) * 6, dict(precision=2, rho_ref=3.0, T_ref=0.06), 0, 0)}


@pytest.mark.parametrize("name", list(CASES))
def test_refreshes_and_states(name):
    from paper_2201_06039_gb300 import lbm
    dims, bc, kw, first, later = CASES[name]
    s, rho, T = _setup(dims, bc)
    lat = _lattice(s, **kw)
    assert lat.kernel == lbm.LBM_KERNEL_FUSED_TMA
    lat.init(rho, T)
    launches = [lbm.lbm_step_profiled(lat.ctx, n)[1] for n in (1, 3)]
    assert launches == [[1, 0, first], [3, 0, later]]
    got = lat.moments()
    lat.close()
    ref = _lattice(s, use_tma=0, **kw)
    ref.init(rho, T)
    ref.step(4)
    want = ref.moments()
    ref.close()
    for k in got:
        assert np.isfinite(got[k]).all()
        assert np.array_equal(got[k], want[k]), k


def test_streamed_frozen_temperature_is_not_refreshed():
    from paper_2201_06039_gb300 import lbm
    s, rho, T = _setup((40, 24, 16), (P, P, P, P, WALL, WALL))
    src = _lattice(s)
    src.init(rho, T)
    src.step(5)
    ckpt = src.save_state()
    src.close()
    lat = _lattice(s, thermal_off=1)
    ref = _lattice(s, thermal_off=1, use_tma=0)
    for start in (lambda x: x.load_state(ckpt), lambda x: x.init(rho, T), lambda x: x.load_state(ckpt)):
        start(lat)
        start(ref)
        n = lbm.lbm_step_profiled(lat.ctx, 4)[1]
        assert n == ([4, 0, 0] if lat.steps_done == 9 else [4, 0, 1]), n
        ref.step(4)
        got, want = lat.moments(), ref.moments()
        for k in got:
            assert np.array_equal(got[k], want[k]), k
    lat.close()
    ref.close()
