"""A stage whose largest speed is exactly zero has no CFL half-step: the march reports
it, whether its half-steps come one by one or many in a launch.  Burgers cells of
+1 and -1 in turn cancel to such a stage after one half-step (the cell averages and,
at P = 1, the point values are exactly zero, the slopes are not)."""
import numpy as np
import pytest

from paper_2104_04347_gb300 import inputs, wcc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [wcc.FP64, wcc.FP32_MIXED])
@pytest.mark.parametrize("calls", [[1] * 4, [4], [2, 2]])
def test_no_half_step_from_a_stage_at_rest(precision, calls):
    q = np.zeros((200, 1, 2))
    q[::2, 0, 0], q[1::2, 0, 0] = 1.0, -1.0
    with wcc.Solver(inputs.BURGERS, 200, 1, (0.0, 1.0), inputs.PERIODIC, precision=precision) as s:
        s.set_initial(q)
        s.step(1, 0.4)
        assert np.all(s.get_dofs()[:, 0, 0] == 0.0)
        s.set_initial(q)
        with pytest.raises(wcc.WCCError) as e:
            for n in calls:
                s.step(n, 0.4)
            s.synchronize()
        assert e.value.code == -5  # WCC_E_NONFINITE
