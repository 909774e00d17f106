"""A frozen-temperature context on a checkpoint of a run with temperature steps on the generic kernel: it
says so, has no plan to report and nothing to autotune, as before such contexts knew the TMA kernel."""
import numpy as np
import pytest

import workloads as W
from tests._parity import inputs

pytestmark = pytest.mark.gpu


def test_streamed_frozen_temperature_reports_the_generic_kernel():
    from paper_2201_06039_gb300 import lbm
    case = W.pool_boiling(40, 24, 32, height=12.0, hot_sigma=4.0)
    s = case["setup"]
    rho, T, _ = (None if a is None else a.astype(np.float32) for a in inputs(case))
    src = lbm.Lattice(lbm.params_from_setup(s))
    src.init(rho, T)
    src.step(3)
    ckpt = src.save_state()
    src.close()
    lat = lbm.Lattice(lbm.params_from_setup(s, thermal_off=1))
    assert lat.kernel == lbm.LBM_KERNEL_FUSED_TMA and lat.plan[0] >= 0
    lat.load_state(ckpt)
    assert lat.kernel == lbm.LBM_KERNEL_FUSED and lat.plan == (-1, 0, 0, 0)
    before = lat.moments()
    with pytest.raises(lbm.LbmError) as e:
        lat.autotune(steps=2)
    assert e.value.status == lbm.LBM_ESTATE
    after = lat.moments()
    for k in before:
        assert np.array_equal(before[k], after[k]), k
    lat.init(rho, T)
    assert lat.kernel == lbm.LBM_KERNEL_FUSED_TMA and lat.plan[0] >= 0
    assert lat.autotune(steps=2)["ms_per_step"] > 0
    lat.close()
