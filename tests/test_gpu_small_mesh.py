"""Meshes that one cluster of CTAs holds: wcc_step takes many half-steps per
launch (at least two per call), and wcc_step(1) the single-half-step kernels.
Both must give the same stage, dt history, time and device state: bit for bit
in FP64 (the same operations), and in FP32-mixed up to the last place of dt (the
cluster forms dt's quotients from a reciprocal), which moves the FP32 coefficients by
a rounding here and there.  Sizes around one tile (127 / 255 new cells), around
powers of two of tiles (the cluster sizes) and at the largest cluster, where the
path ends."""
import numpy as np
import pytest

from paper_2104_04347_gb300 import inputs, wcc

pytestmark = pytest.mark.gpu

CFL = {1: 0.4, 2: 0.3, 3: 0.25, 4: 0.2, 5: 0.16, 6: 0.14}


def _problem(system, N, P, bc):
    if system == inputs.EULER:
        pr = inputs.euler_density_wave(N, P)
        return pr.q0 if bc == inputs.PERIODIC else np.concatenate([pr.q0, pr.q0[:1]])
    if system == inputs.BURGERS:
        q = inputs.burgers_fourier(N, P).q0
    else:
        q = inputs.advection_sine(N, P, 0.0, 1.0).q0
    return q if bc == inputs.PERIODIC else np.concatenate([q, q[:1]])


def _run(system, N, P, bc, precision, calls):
    with wcc.Solver(system, N, P, (0.0, 1.0), bc, precision=precision) as s:
        s.set_initial(_problem(system, N, P, bc))
        for n in calls:
            s.step(n, CFL[P])
        return s.get_dofs(), s.dt_history(), s.state(), s.launch_count()


SIZES = {wcc.FP64: [4, 127, 128, 254, 509, 2031, 2032, 2033], wcc.FP32_MIXED: [4, 255, 256, 510, 1021, 4079, 4080, 4081]}


@pytest.mark.parametrize("precision,N", [(p, n) for p in SIZES for n in SIZES[p]])
@pytest.mark.parametrize("bc", [inputs.PERIODIC, inputs.TRANSMISSIVE])
@pytest.mark.parametrize("system,P", [(inputs.EULER, 3), (inputs.BURGERS, 4), (inputs.ADVECTION, 1)])
def test_cluster_equals_single_half_steps(precision, N, bc, system, P):
    got, want = _run(system, N, P, bc, precision, [3, 8, 1, 4]), _run(system, N, P, bc, precision, [1] * 16)
    assert got[2][1:] == want[2][1:] == (16, 0)
    if precision == wcc.FP64:
        assert np.array_equal(got[1], want[1]) and np.array_equal(got[0], want[0]) and got[2] == want[2]
    else:
        assert np.allclose(got[1], want[1], rtol=5e-16, atol=0.0)
        # averages carry 48 bits, coefficients 24: a last-place change of dt moves
        # them by a few units of their last place
        assert np.max(np.abs(got[0][..., 0] - want[0][..., 0])) <= 1e-9
        assert np.max(np.abs(got[0] - want[0])) <= 1e-5 * np.max(np.abs(want[0]))
    cells = N + 1 if bc == inputs.TRANSMISSIVE else N
    if cells <= (2032 if precision == wcc.FP64 else 4080):  # fewer launches than half-steps: the cluster ran
        assert got[3] < want[3]


@pytest.mark.parametrize("P", [5, 6])
def test_cluster_high_order(P):
    got = _run(inputs.EULER, 300, P, inputs.PERIODIC, wcc.FP64, [7, 6])
    want = _run(inputs.EULER, 300, P, inputs.PERIODIC, wcc.FP64, [1] * 13)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


def test_more_half_steps_than_one_launch_takes():
    got = _run(inputs.BURGERS, 130, 2, inputs.PERIODIC, wcc.FP64, [531])
    want = _run(inputs.BURGERS, 130, 2, inputs.PERIODIC, wcc.FP64, [1] * 531)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]) and got[2] == want[2]


def test_errors_are_reported():
    q = _problem(inputs.EULER, 200, 2, inputs.PERIODIC)
    q[100, 2, 1] = 1e3  # a slope that makes the pressure negative after a half-step
    with wcc.Solver(inputs.EULER, 200, 2, (0.0, 1.0), inputs.PERIODIC) as s:
        s.set_initial(q)
        s.step(20, 0.3)
        with pytest.raises(wcc.WCCError) as e:
            s.synchronize()
        assert e.value.code in (-5, -6)
