"""The TMA kernel on lattices with walls, outflow and thermal faces across x and y and with a frozen
temperature: step after step it computes exactly what the generic fused and the two-pass kernels
compute (the pulls past a face are patched from the staged window there, and read through wrapped or
clamped coordinates here).  Also small z-chunks, and read-out calls with some of the outputs."""
import numpy as np
import pytest

import workloads as W
from tests._parity import inputs, run_gpu

pytestmark = pytest.mark.gpu

P, WALL, OUT, TH = W.BC_PERIODIC, W.BC_WALL, W.BC_OUTFLOW, W.BC_THERMAL_ONLY
FACES = {"box": (WALL,) * 6, "walls_x": (WALL, WALL, P, P, WALL, OUT), "open_x_walls_y": (OUT, OUT, WALL, WALL, WALL, WALL),
         "wall_outflow_x": (WALL, OUT, P, P, P, P), "outflow_wall_y": (P, P, OUT, WALL, OUT, WALL),
         "all_open": (OUT,) * 6, "corners": (WALL, OUT, OUT, WALL, WALL, OUT), "thermal_x_walls_y": (TH, TH, WALL, WALL, P, P)}


def _case(dims, bc, **kw):
    nx, ny, nz = dims
    s = W.LatticeSetup(nx, ny, nz, bc=bc, T_wall_over_Tc=(0.86, 0.87, 0.865, 0.855, 0.88, 0.86), sigma=W.SIGMA_STAR,
                       gravity=(1e-6, 0, -3e-5), hot_dT_over_Tc=0.05, hot_sigma=4.0, **kw)
    case = dict(name=f"{dims} {bc}", setup=s, kind="pool", height=nz / 2.0, W=4.0, Tr_liquid=0.86, noise=1e-3,
                noise_seed=W.MASTER_SEED + nx)
    return case


def _compare(case, steps, **over):
    from paper_2201_06039_gb300 import lbm
    s = case["setup"]
    rho, T, u = inputs(case)
    lat = lbm.Lattice(lbm.params_from_setup(s, kernel=2, use_tma=1, **over))
    assert lat.kernel == lbm.LBM_KERNEL_FUSED_TMA
    lat.close()
    tma, _ = run_gpu(s, rho, T, u, steps, kernel=2, use_tma=1, **over)
    gen, _ = run_gpu(s, rho, T, u, steps, kernel=2, use_tma=0, **over)
    two, _ = run_gpu(s, rho, T, u, steps, kernel=1, **over)
    for k in tma:
        assert np.isfinite(tma[k]).all()
        assert np.array_equal(tma[k], gen[k]), k
        assert np.array_equal(tma[k], two[k]), k


@pytest.mark.parametrize("faces", list(FACES))
@pytest.mark.parametrize("dims", [(4, 4, 5), (37, 11, 19), (50, 45, 9), (88, 49, 12)])
def test_tma_faces_bit_identical(dims, faces):
    _compare(_case(dims, FACES[faces]), 7)


@pytest.mark.parametrize("faces", ["box", "corners", "walls_x"])
@pytest.mark.parametrize("precision", [1, 2])
def test_tma_faces_16bit_bit_identical(faces, precision):
    _compare(_case((41, 19, 14), FACES[faces]), 7, precision=precision, rho_ref=3.0, T_ref=0.06)


@pytest.mark.parametrize("faces", ["box", "corners", "periodic"])
@pytest.mark.parametrize("dims", [(41, 27, 15), (48, 40, 9)])
@pytest.mark.parametrize("wet", [False, True])
def test_tma_frozen_temperature_bit_identical(dims, faces, wet):
    bc = FACES.get(faces, (P, P, P, P, WALL, WALL))
    kw = dict(wall_scheme=1, wall_phi=1.1, wall_drho=0.05) if wet else {}
    _compare(_case(dims, bc, thermal_off=1, **kw), 7)


def test_frozen_temperature_resumes_from_an_evolving_run():
    """A checkpoint of a run with temperature holds g in streamed form: a frozen-temperature context
    that loads it must take the generic kernel, and gives the same state either way."""
    from paper_2201_06039_gb300 import lbm
    case = _case((40, 24, 16), (P, P, P, P, WALL, WALL))
    s = case["setup"]
    rho, T, _ = inputs(case)
    src = lbm.Lattice(lbm.params_from_setup(s))
    src.init(rho.astype(np.float32), T.astype(np.float32))
    src.step(5)
    ckpt = src.save_state()
    src.close()
    out = []
    for tma in (0, 1):
        lat = lbm.Lattice(lbm.params_from_setup(s, kernel=2, use_tma=tma, thermal_off=1))
        lat.load_state(ckpt)
        lat.step(6)
        out.append(lat.moments())
        lat.close()
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]), k


@pytest.mark.parametrize("zchunk", [1, 2, 3, 0])
def test_small_z_chunks_bit_identical(zchunk):
    from paper_2201_06039_gb300 import lbm
    case = _case((33, 20, 11), (P, P, P, P, WALL, OUT))
    s = case["setup"]
    rho, T, u = inputs(case)
    gen, _ = run_gpu(s, rho, T, u, 9, kernel=2, use_tma=0)
    lat = lbm.Lattice(lbm.params_from_setup(s, kernel=2, use_tma=1))
    lat.select_plan(-1, zchunk)
    lat.init(rho.astype(np.float32), T.astype(np.float32))
    lat.step(9)
    m = lat.moments()
    lat.close()
    for k in m:
        assert np.array_equal(m[k], gen[k]), (zchunk, k)


@pytest.mark.parametrize("dims", [(1, 1, 3), (33, 9, 5), (64, 17, 40)])
def test_readout_of_some_fields_host_and_device(dims):
    import torch
    from paper_2201_06039_gb300 import lbm
    case = _case(dims, (P, P, P, P, P, P))
    s = case["setup"]
    rho, T, _ = inputs(case)
    lat = lbm.Lattice(lbm.params_from_setup(s))
    lat.init(rho.astype(np.float32), T.astype(np.float32))
    lat.step(3)
    ref = lat.moments()
    dev = torch.full(lat.shape, -1.0, device="cuda")
    host = np.full(lat.shape, -1.0, dtype=np.float32)
    lbm.lbm_get_moments(lat.ctx, rho=dev, uz=host)
    assert np.array_equal(dev.cpu().numpy(), ref["rho"]) and np.array_equal(host, ref["uz"])
    mass, tsum, _ = lat.totals()
    assert abs(mass - ref["rho"].astype(np.float64).sum()) <= 1e-12 * mass
    lat.close()
