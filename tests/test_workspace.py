"""Workspace of a context: the (psi, rho) field, 8 bytes a node, only where a kernel reads it."""
import pytest

from paper_2201_06039_gb300 import lbm


def _bytes(dims, **kw):
    p = lbm.lbm_params_default()
    p.nx, p.ny, p.nz = dims
    for k, v in kw.items():
        setattr(p, k, v)
    return lbm.lbm_workspace_bytes(p)


@pytest.mark.parametrize("kw", [{}, dict(precision=1), dict(thermal_q=19), dict(flow_off=1), dict(thermal_off=1)])
@pytest.mark.parametrize("dims", [(200, 200, 300), (64, 64, 96), (33, 9, 17), (64, 64, 2)])
def test_fused_contexts_hold_no_psi_field(dims, kw):
    n = dims[0] * dims[1] * dims[2]
    field = (8 * n + 255) // 256 * 256
    two = _bytes(dims, kernel=1, **kw)
    assert _bytes(dims, kernel=2, **kw) == two - field
    assert _bytes(dims, kernel=0, **kw) == two - field


@pytest.mark.parametrize("dims", [(300, 300, 1), (256, 256, 1), (200, 200, 3)])
def test_thin_lattices_read_out_through_it(dims):
    assert _bytes(dims, kernel=2) == _bytes(dims, kernel=1)


def test_finite_difference_divu_runs_the_two_pass_kernels():
    assert _bytes((64, 64, 96), divu_mode=1, kernel=0) == _bytes((64, 64, 96), divu_mode=1, kernel=1)
