"""lbm_get_moments runs the TMA kernel's read-out on larger lattices, whose waits are bounded: when one
gives up the call reports LBM_ETIMEOUT (the fields it wrote are not those of the state), and the state, the
next read-out and the next step are as if it had not been made."""
import numpy as np
import pytest

import workloads as W
from tests._parity import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("check", [0, 1])
@pytest.mark.parametrize("use_graph", [0, 1])
def test_a_readout_wait_that_gives_up_is_reported(check, use_graph):
    from paper_2201_06039_gb300 import lbm
    case = W.pool_boiling(64, 48, 48, height=20.0, hot_sigma=4.0)     # 147456 nodes: read out by the TMA kernel
    s = case["setup"]
    rho, T, _ = inputs(case)

    def run(stall):
        lat = lbm.Lattice(lbm.params_from_setup(s, check_nonfinite=check, use_graph=use_graph, test_stall=stall))
        assert lat.kernel == lbm.LBM_KERNEL_FUSED_TMA
        lat.init(rho.astype(np.float32), T.astype(np.float32))
        lat.step(4)
        if stall:
            with pytest.raises(lbm.LbmError) as e:
                lat.moments()
            assert e.value.status == lbm.LBM_ETIMEOUT
        m = [lat.moments()]
        lat.step(3)
        m.append(lat.moments())
        lat.close()
        return m

    got, want = run(2), run(0)
    for a, b in zip(got, want):
        for k in a:
            assert np.isfinite(a[k]).all()
            assert np.array_equal(a[k], b[k]), k
