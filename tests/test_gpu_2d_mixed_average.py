"""The FP32-mixed 2D stage keeps the cell average to the 48 bits of its two floats and
the conversions lose no more: a point value loaded and read back, with coefficients
that 24 bits hold exactly, returns within 1.25 x 2^-49 of its size and its even
correction's together.  (The low float is below 2^-24 of the average's power of two,
half its last place 2^-49; the FP64 sums round four times, 2^-53 each.)"""
import numpy as np
import pytest

from paper_2104_04347_gb300 import inputs, wcc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [1, 2, 3])
@pytest.mark.parametrize("size", [1e-3, 1.0, 30.0])
def test_average_there_and_back(P, size):
    rng = np.random.default_rng(10 * P)
    nq = (P + 1) * (P + 2) // 2
    fact = np.array([1, 1, 1, 2, 1, 2, 6, 2, 2, 6][:nq], dtype=np.float64)
    q = (size * rng.standard_normal((64, 200, 1, nq))).astype(np.float32).astype(np.float64) * fact
    q[..., 0] = 1.0 + 0.3 * rng.standard_normal((64, 200, 1))
    with wcc.Solver2D(inputs.ADVECTION, 200, 64, P, (0.0, 1.0, 0.0, 1.0), inputs.PERIODIC, precision=wcc.FP32_MIXED) as s:
        s.set_initial(q)
        back = s.get_dofs()
    corr = np.abs(q[..., 3]) / 24 + np.abs(q[..., 5]) / 24 if P >= 2 else 0.0
    assert np.array_equal(back[..., 1:], q[..., 1:])
    assert np.max(np.abs(back[..., 0] - q[..., 0]) / (np.abs(q[..., 0]) + corr)) <= 1.25 * 2.0 ** -49
