"""cells_per_block and graph_chunk act on meshes that one cluster of CTAs would hold:
a tile size, or graph_chunk = 0, takes the one-half-step kernels (one launch per
half-step in the launch count), the defaults take the cluster, and the results are the
same bits.  The tuner has the cluster among its candidates there and keeps what it chose."""
import numpy as np
import pytest

from paper_2104_04347_gb300 import inputs, wcc

pytestmark = pytest.mark.gpu


def _run(precision, N, P, **options):
    pr = inputs.euler_density_wave(N, P)
    with wcc.Solver(pr.system, N, P, (pr.x_l, pr.x_r), pr.bc, precision=precision, **options) as s:
        s.set_initial(pr.q0)
        before = s.launch_count()
        s.step(64, 0.2)
        return s.get_dofs(), s.dt_history(), s.launch_count() - before - 1  # less the read-back


@pytest.mark.parametrize("precision,N,P,options", [
    (wcc.FP64, 1000, 3, {"cells_per_block": 127}), (wcc.FP64, 1000, 3, {"graph_chunk": 0}), (wcc.FP64, 300, 5, {"graph_chunk": 0}),
    (wcc.FP32_MIXED, 1607, 2, {"cells_per_block": 255}), (wcc.FP32_MIXED, 1607, 2, {"cells_per_block": 510}),
    (wcc.FP32_MIXED, 1607, 3, {"cells_per_block": 255}), (wcc.FP32_MIXED, 1607, 3, {"cells_per_block": 510}),
    (wcc.FP32_MIXED, 1607, 4, {"graph_chunk": 0})])
def test_options_act(precision, N, P, options):
    q, dts, launches = _run(precision, N, P)
    assert launches == 1
    got, got_dts, got_launches = _run(precision, N, P, **options)
    assert got_launches == 64
    assert np.array_equal(got_dts, dts) and np.array_equal(got, q)


def test_tuner_on_a_small_mesh():
    pr = inputs.euler_density_wave(1000, 3)
    with wcc.Solver(pr.system, 1000, 3, (pr.x_l, pr.x_r), pr.bc, precision=wcc.FP32_MIXED) as s:
        s.set_initial(pr.q0)
        chosen = s.autotune(0.2)
        assert chosen in [(0, 1), (255, 1), (510, 1), (0, 2)]
        assert np.array_equal(s.dt_history(), [])
        before = s.launch_count()
        s.step(64, 0.2)
        n = s.launch_count() - before
    assert n == 1 if chosen == (0, 1) else n >= 32
