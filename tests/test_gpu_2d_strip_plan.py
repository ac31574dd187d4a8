"""The strip height and width picked from the mesh (rows_per_cta = 16, the
default) only change how a half-step is split among CTAs: the stage equals,
bit for bit, that of full-width strips of a given height, at meshes of one
strip or less, around multiples of the strip widths (31, 63, 95 and 127 new
columns) and with strips of every remainder."""
import numpy as np
import pytest

from paper_2104_04347_gb300 import inputs, wcc
from tests.test_gpu_2d import ADV, CFL, EULER, _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [wcc.FP64, wcc.FP32_MIXED, wcc.FP32])
@pytest.mark.parametrize("system,P", [(EULER, 3), (EULER, 1), (ADV, 2)])
@pytest.mark.parametrize("bc", [inputs.PERIODIC, inputs.TRANSMISSIVE])
@pytest.mark.parametrize("nx,ny", [(4, 5), (31, 9), (63, 33), (128, 65), (190, 70)])
def test_picked_strips_equal_given_ones(precision, system, P, bc, nx, ny):
    pr = _problem(ADV, nx, ny, P, bc)
    if system == EULER:  # a density wave in uniform flow, physical on any mesh
        rho = 0.2 * pr.q0[:, :, 0]
        rho[..., 0] += 1.0
        E = 0.5 * (0.5 ** 2 + 0.3 ** 2) * rho
        E[..., 0] += 1.0 / 0.4
        pr.q0 = np.stack([rho, 0.5 * rho, -0.3 * rho, E], axis=2)
    got = []
    for rows in (16, 7):
        with wcc.Solver2D(system, nx, ny, P, (pr.x_l, pr.x_r, pr.y_l, pr.y_r), bc, precision=precision, ax=pr.ax,
                          ay=pr.ay, rows_per_cta=rows) as s:
            s.set_initial(pr.q0)
            s.step(3, 0.5 * CFL[P])
            got.append((s.get_dofs(), s.dt_history()))
    assert np.array_equal(got[0][1], got[1][1])
    assert np.array_equal(got[0][0], got[1][0])
