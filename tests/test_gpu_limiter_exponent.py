"""Limiter exponents other than 2 (the option alpha): data with a jump, half-step by
half-step against the oracle from the stage the GPU holds, in FP64 and FP32-mixed,
1D below and above the size one cluster of CTAs marches (whose marches must give
the bits of single half-steps) and 2D.  Bounds as for alpha = 2: FP64 1e-11 of a
variable's scale or 50 x the oracle's spread under 4e-16 noise (tests/gpu_common.py),
FP32-mixed 2e-6 or 50 x the spread under 1e-7 (2D: in L1, 2e-7)."""
import numpy as np
import pytest

import oracle
from paper_2104_04347_gb300 import inputs, wcc
from tests.gpu_common import SCATTER_FACTOR, TOL64, scales

pytestmark = pytest.mark.gpu

CFL = {1: 0.4, 3: 0.25}


def _worst(got, ref, q, half, noise, floor):
    rng = np.random.default_rng(5)
    spread = np.zeros_like(ref)
    for _ in range(3):
        spread = np.maximum(spread, np.abs(half(q * (1.0 + noise * rng.standard_normal(q.shape))) - ref))
    bound = np.maximum(floor * scales(ref)[None, :, None], SCATTER_FACTOR * spread)
    return float(np.max(np.abs(got - ref) / bound))


@pytest.mark.parametrize("alpha", [1.0, 3.0])
@pytest.mark.parametrize("P", [1, 3])
@pytest.mark.parametrize("precision,N", [(wcc.FP64, 300), (wcc.FP64, 2100), (wcc.FP32_MIXED, 300), (wcc.FP32_MIXED, 4200)])
def test_1d(precision, N, P, alpha):
    pr = inputs.euler_riemann_seeded(N, P)
    law = oracle.make_law(pr.system, P, bc=pr.bc, alpha=alpha)
    noise, floor = (4e-16, TOL64) if precision == wcc.FP64 else (1e-7, 2e-6)
    with wcc.Solver(pr.system, N, P, (pr.x_l, pr.x_r), pr.bc, precision=precision, alpha=alpha) as s:
        s.set_initial(pr.q0)
        prev = s.get_dofs()
        for n in range(12):
            s.step(1, CFL[P])
            cur, lam = s.get_dofs(), s.dt_history()[-1] / pr.dx
            half = lambda q: oracle.halfstep(law, n & 1, q, lam)
            assert _worst(cur, half(prev), prev, half, noise, floor) <= 1.0, n
            prev = cur
        one_by_one, dts = prev, s.dt_history()
        s.set_initial(pr.q0)
        s.step(12, CFL[P])
        assert np.array_equal(s.get_dofs(), one_by_one) and np.array_equal(s.dt_history(), dts)


@pytest.mark.parametrize("alpha", [1.0, 3.0])
@pytest.mark.parametrize("P", [1, 3])
@pytest.mark.parametrize("precision", [wcc.FP64, wcc.FP32_MIXED])
def test_2d(precision, P, alpha):
    pr = inputs.riemann2d(40, P)
    law = oracle.make_law2d(pr.system, P, bc=pr.bc, alpha=alpha)
    rng = np.random.default_rng(6)
    with wcc.Solver2D(pr.system, 40, 40, P, (pr.x_l, pr.x_r, pr.y_l, pr.y_r), pr.bc, precision=precision, alpha=alpha) as s:
        s.set_initial(pr.q0)
        prev = s.get_dofs()
        for n in range(6):
            s.step(1, CFL[P])
            cur, dt = s.get_dofs(), s.dt_history()[-1]
            half = lambda q: oracle.halfstep2d(law, n & 1, q, dt / pr.dx, dt / pr.dy)
            ref = half(prev)
            sc = np.max(np.abs(ref[..., 0]), axis=(0, 1))
            noise = 4e-16 if precision == wcc.FP64 else 1e-7
            moved = [np.abs(half(prev * (1.0 + noise * rng.standard_normal(prev.shape))) - ref) for _ in range(3)]
            if precision == wcc.FP64:
                bound = np.maximum(TOL64 * sc[None, None, :, None], SCATTER_FACTOR * np.maximum.reduce(moved))
                assert np.max(np.abs(cur - ref) / bound) <= 1.0, n
            else:
                l1 = lambda a: np.mean(a, axis=(0, 1, 3)) / sc
                bound = np.maximum(2e-7, SCATTER_FACTOR * np.maximum.reduce([l1(m) for m in moved]))
                assert np.all(l1(np.abs(cur - ref)) <= bound), n
            prev = cur
