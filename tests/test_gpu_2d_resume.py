"""A 2D FP64 run that is stopped (wcc2d_get_dofs) and resumed from what was read back
(wcc2d_set_initial in a new handle) goes on bit for bit, and loading any stage and
reading it back returns its bits: every value is kept so that the conversion there
and back is exact."""
import numpy as np
import pytest

from paper_2104_04347_gb300 import inputs, wcc
from tests.test_gpu_2d import ADV, CFL, EULER, _problem

pytestmark = pytest.mark.gpu


def _solver(system, nx, ny, P, pr, bc):
    return wcc.Solver2D(system, nx, ny, P, (pr.x_l, pr.x_r, pr.y_l, pr.y_r), bc, ax=pr.ax, ay=pr.ay)


@pytest.mark.parametrize("P", [1, 2, 3])
@pytest.mark.parametrize("system", [ADV, EULER])
@pytest.mark.parametrize("bc", [inputs.PERIODIC, inputs.TRANSMISSIVE])
def test_resumed_run_equals_uninterrupted(system, P, bc):
    nx, ny = 45, 38
    pr = _problem(ADV, nx, ny, P, bc)
    if system == EULER:  # a density wave in uniform flow
        rho = 0.2 * pr.q0[:, :, 0]
        rho[..., 0] += 1.0
        E = 0.5 * (0.5 ** 2 + 0.3 ** 2) * rho
        E[..., 0] += 1.0 / 0.4
        pr.q0 = np.stack([rho, 0.5 * rho, -0.3 * rho, E], axis=2)
    with _solver(system, nx, ny, P, pr, bc) as s:
        s.set_initial(pr.q0)
        s.step(8, 0.5 * CFL[P])
        middle = s.get_dofs()
        s.step(6, 0.5 * CFL[P])
        want, dts = s.get_dofs(), s.dt_history()
    with _solver(system, nx, ny, P, pr, bc) as s:
        s.set_initial(middle)
        assert np.array_equal(s.get_dofs(), middle)
        s.step(6, 0.5 * CFL[P])
        assert np.array_equal(s.dt_history(), dts[8:])
        assert np.array_equal(s.get_dofs(), want)


@pytest.mark.parametrize("P", [1, 2, 3])
def test_any_stage_comes_back(P):
    rng = np.random.default_rng(P)
    q = rng.standard_normal((33, 70, 4, (P + 1) * (P + 2) // 2)) * 10.0 ** rng.uniform(-12, -2, (33, 70, 4, (P + 1) * (P + 2) // 2))
    q[..., 0] += np.array([1.0, 0.3, -0.2, 3.0])
    with wcc.Solver2D(inputs.EULER, 70, 33, P, (0.0, 1.0, 0.0, 1.0), inputs.PERIODIC) as s:
        s.set_initial(q)
        assert np.array_equal(s.get_dofs(), q)
