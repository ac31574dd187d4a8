"""wcc_step_until on meshes one cluster of CTAs marches, with a varying speed: the same
dt list, stage and step count as with a launch per half-step (graph_chunk = 0), bit
for bit, for end times that cut a pair of half-steps in two (the cluster stops on a
half stage and the host takes the rest) and ones that do not."""
import numpy as np
import pytest

from paper_2104_04347_gb300 import inputs, wcc

pytestmark = pytest.mark.gpu


def _solver(pr, precision, **options):
    return wcc.Solver(pr.system, pr.N, pr.P, (pr.x_l, pr.x_r), pr.bc, precision=precision, **options)


def _until(pr, precision, t_end, **options):
    with _solver(pr, precision, **options) as s:
        s.set_initial(pr.q0)
        taken = s.step_until(t_end, 0.2)
        return s.get_dofs(), s.dt_history(), s.state(), taken


@pytest.mark.parametrize("precision", [wcc.FP64, wcc.FP32_MIXED])
@pytest.mark.parametrize("make", [lambda: inputs.euler_riemann_seeded(300, 3), lambda: inputs.euler_riemann_seeded(700, 2),
                                  lambda: inputs.burgers_fourier(500, 3)], ids=["euler300", "euler700", "burgers500"])
@pytest.mark.parametrize("cut", [True, False])
def test_cluster_march_to_a_time(make, precision, cut):
    pr = make()
    with _solver(pr, precision) as s:
        s.set_initial(pr.q0)
        s.step(400, 0.2)
        d = s.dt_history()
    if cut:  # where the step grows most within a pair, end a little before the pair's end
        m = 10 + int(np.argmax(d[21::2][:150] / d[20::2][:150]))
        growth = d[2 * m + 1] / d[2 * m] - 1.0
        assert growth > 1e-11  # well above the rule's slack of 1e-12
        t_end = float(np.sum(d[:2 * m + 1])) + d[2 * m + 1] * (1.0 - 0.5 * growth)
    else:
        m = 150
        t_end = float(np.sum(d[:2 * m])) + 0.7 * d[2 * m]
    got, want = _until(pr, precision, t_end), _until(pr, precision, t_end, graph_chunk=0)
    assert np.array_equal(got[1], want[1]) and np.array_equal(got[0], want[0]) and got[2:] == want[2:]
    q, dts, (t, steps, parity), taken = got
    assert parity == 0 and taken == steps == 2 * m + 2 and abs(t - t_end) <= 1e-12
    assert np.array_equal(dts[:2 * m + (1 if cut else 0)], d[:2 * m + (1 if cut else 0)])
    if cut:
        assert dts[-1] < d[2 * m + 1] and dts[-2] == d[2 * m]
    else:
        assert dts[-1] == dts[-2]
