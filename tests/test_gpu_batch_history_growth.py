"""The dt histories of a batch grow while it marches: captured launches are taken
again for the new buffer.  A batch in pairs that passes the first capacity (1024
half-steps) between calls has the dt lists and stages of one that marched in a
single call."""
import numpy as np
import pytest

from paper_2104_04347_gb300 import inputs, wcc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth", [1, 2])
def test_march_past_the_first_capacity(depth):
    members = [inputs.euler_density_wave(300, 2), inputs.euler_density_wave(520, 3)]
    got = []
    for calls in ([960, 128, 96], [1184]):
        with wcc.Batch(members, tb_depth=depth) as b:
            b.set_initial()
            for n in calls:
                b.step(n, 0.2)
            got.append((b.get_dofs(), [b.dt_history(i) for i in range(2)], b.state()))
    assert got[0][2] == got[1][2] == (1184, 0)
    for i in range(2):
        assert len(got[0][1][i]) == 1184 and np.all(got[0][1][i] > 0.0)
        assert np.array_equal(got[0][1][i], got[1][1][i]) and np.array_equal(got[0][0][i], got[1][0][i])
