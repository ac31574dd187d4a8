"""How half-steps are grouped into calls leaves no trace: FP32-mixed meshes that one
cluster of CTAs holds give, for wcc_step(3), (8), (1), (4), the bits of sixteen calls of
wcc_step(1), which take the single-half-step kernels (FP64: test_gpu_small_mesh).
Shock tubes too: behind a jump the limiter acts on one characteristic component
and not on the others."""
import numpy as np
import pytest

from paper_2104_04347_gb300 import inputs, wcc
from tests.test_gpu_reproducible import CFL, _sine, _tube, _wave

pytestmark = pytest.mark.gpu


def _run(system, N, P, bc, q, calls):
    with wcc.Solver(system, N, P, (0.0, 1.0), bc, precision=wcc.FP32_MIXED) as s:
        s.set_initial(q)
        for n in calls:
            s.step(n, CFL[P])
        return s.get_dofs(), s.dt_history(), s.state(), s.launch_count()


@pytest.mark.parametrize("N", [4, 255, 256, 1021, 4079])
@pytest.mark.parametrize("P", [1, 2, 3, 4])
@pytest.mark.parametrize("data", ["wave", "tube", "burgers"])
def test_mixed_cluster_equals_single_half_steps(N, P, data):
    system = inputs.BURGERS if data == "burgers" else inputs.EULER
    bc = inputs.TRANSMISSIVE if data == "tube" else inputs.PERIODIC
    q = _tube(N, P) if data == "tube" else _wave(N, P, 0.7, bc) if data == "wave" else _sine(N, P, 0.25, 0.7, 0.5)
    got, want = _run(system, N, P, bc, q, [3, 8, 1, 4]), _run(system, N, P, bc, q, [1] * 16)
    assert np.array_equal(got[1], want[1]) and np.array_equal(got[0], want[0]) and got[2] == want[2]
    assert got[3] < want[3]  # the cluster ran
