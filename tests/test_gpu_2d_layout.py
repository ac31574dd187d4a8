"""The 2D layout conversions (host scaled derivatives <-> planes of Taylor
coefficients) move every value to its place and back: loading a stage and
reading it back returns it up to the rounding of the storage, on meshes around
the conversion's tile of 64 cells, for every degree, number of variables and
precision.  Bounds: FP64 rounds twice per value (by 1/(k! l!) and back), FP32
once to 24 bits; FP32-mixed keeps the point value to the float-float average's
46 bits of the largest term."""
import numpy as np
import pytest

from paper_2104_04347_gb300 import inputs, wcc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [wcc.FP64, wcc.FP32, wcc.FP32_MIXED])
@pytest.mark.parametrize("P", [1, 2, 3])
@pytest.mark.parametrize("system", [inputs.ADVECTION, inputs.EULER])
@pytest.mark.parametrize("nx,ny,bc", [(4, 4, inputs.PERIODIC), (63, 5, inputs.TRANSMISSIVE), (64, 6, inputs.PERIODIC),
                                      (65, 7, inputs.PERIODIC), (191, 4, inputs.TRANSMISSIVE)])
def test_load_and_read_back(precision, P, system, nx, ny, bc):
    rng = np.random.default_rng(1000 * P + nx)
    cy, cx = (ny, nx) if bc == inputs.PERIODIC else (ny + 1, nx + 1)
    nv, nq = (4 if system == inputs.EULER else 1), (P + 1) * (P + 2) // 2
    q = 0.01 * rng.standard_normal((cy, cx, nv, nq))
    q[..., 0] += np.arange(1, nv + 1) if system == inputs.ADVECTION else np.array([1.0, 0.3, -0.2, 3.0])
    q[0, 0, 0, nq - 1] = 0.0
    with wcc.Solver2D(system, nx, ny, P, (0.0, 1.0, 0.0, 1.0), bc, precision=precision) as s:
        s.set_initial(q)
        back = s.get_dofs()
    d = np.abs(back - q)
    if precision == wcc.FP64:
        assert np.all(d <= 2.0 ** -52 * np.abs(q))
        return
    assert np.all(d[..., 1:] <= 2.0 ** -23 * np.abs(q[..., 1:]))
    if precision == wcc.FP32:
        assert np.all(d[..., 0] <= 2.0 ** -24 * np.abs(q[..., 0]))
    else:
        # the average's corrections come from the coefficients before and after
        # their rounding to 24 bits, a twelfth of it at most
        corr = np.abs(q[..., 3]) + np.abs(q[..., 5]) if P >= 2 else 0.0
        assert np.all(d[..., 0] <= 2.0 ** -45 * np.abs(q[..., 0]) + 2.0 ** -24 / 12 * corr)
