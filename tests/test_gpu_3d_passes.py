"""The two-pass 3-D FV step (the default on small FP32 grids the staged flux
passes serve) against the four staged passes: equal populations, bit for bit, over
calls of one and of several steps, on periodic and walled z, blocks with a
ragged edge on y and z, and axes shorter than the stencil."""
import numpy as np
import pytest

from tests import inputs
from tests.test_gpu_3d import STAGED_CASES, _ids, _params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", STAGED_CASES + [dict(nx=128, ny=9, nz=7, bcz=1, thermal=True)], ids=_ids)
def test_two_passes_match_the_staged(lbgpu, case):
    lb, th = lbgpu, case.get("thermal", False)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    f = inputs.random_populations3(nx, ny, nz, seed=3 * nx + nz, amp=0.2)
    t = inputs.random_populations3(nx, ny, nz, seed=9, amp=0.2) if th else None
    out = []
    for sched in (lb.LB3_FV_STAGED, lb.LB3_FV_AUTO):
        g = lb.Grid3(**case, store=lb.LB_STORE_F32).init(**_params(th)).set_fv_schedule(sched)
        out.append(g.set_pops(f, t).step_fv(1).step_fv(3).get_pops())
    assert np.array_equal(out[0][0], out[1][0])
    assert not th or np.array_equal(out[0][1], out[1][1])
