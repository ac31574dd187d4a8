"""1D marches give the same bits as ever: SHA-256 digests of the stage and the dt list
of marches recorded on a GB300 from the library as its kernels first were
(tests/golden/fp64_marches_1d.txt, mixed_marches_1d.txt), for every system, degree,
boundary, limiter option and route (one cluster of CTAs, single half-steps on larger
meshes, FP32-mixed also two half-steps per launch and batches).

Bits, because no tolerance would do: where a one-sided slope of the limiter nearly
vanishes, or behind a shock, the scheme multiplies rounding, and after some hundred
half-steps two ways of rounding the same formulas differ by 1e-5 (a smooth sine)
or by O(1) (a shock tube to t = 0.05).  The data are formed with additions and
multiplications only, so that every machine hands over the same ones."""
import hashlib
import os

import numpy as np
import pytest

from paper_2104_04347_gb300 import inputs, wcc

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")
CFL = {1: 0.4, 2: 0.3, 3: 0.25, 4: 0.22, 5: 0.16, 6: 0.14}


def _cos_sin(t):
    c = s = 0.0
    term = 1.0
    for k in range(40):
        if k % 2 == 0:
            c += term if k % 4 == 0 else -term
        else:
            s += term if k % 4 == 1 else -term
        term = term * t / (k + 1)
    return c, s


def _sine(N, P, amp, phase, mean=0.0):
    """Point values and scaled derivatives of mean + amp sin(pi x + phase) on N cells of [0, 2)."""
    d = 2.0 * 3.141592653589793 / N
    (cd, sd), (c, s) = _cos_sin(d), _cos_sin(phase)
    q = np.zeros((N, 1, P + 1))
    for i in range(N):
        f = amp
        for k in range(P + 1):
            q[i, 0, k] = f * (s, c, -s, -c)[k % 4]
            f = f * d
        q[i, 0, 0] += mean
        c, s = c * cd - s * sd, s * cd + c * sd
    return q


def _wave(N, P, phase, bc):
    d = _sine(N, P, 0.15, phase)[:, 0]
    if bc == inputs.TRANSMISSIVE:
        d = np.concatenate([d, d[:1]])
    d[:, 0] += 1.0
    u, p = 0.75, 0.9
    q = np.stack([d, u * d, 0.5 * u * u * d], axis=1)
    q[:, 2, 0] += p / 0.4
    return q


def _tube(N, P):
    q = np.zeros((N + 1, 3, P + 1))
    for i in range(N + 1):
        f = min(max(0.5 * N - (i - 0.5), 0.0), 1.0)
        for v, (l, r) in enumerate(((1.0, 0.375), (0.25, -0.125), (2.5, 0.75))):
            q[i, v, 0] = f * l + (1.0 - f) * r
    return q


def marches():
    """name -> (system, N, P, domain, bc, data, ("until", t) or ("step", n), options)"""
    out = {}
    A, B, E, PER, TR = inputs.ADVECTION, inputs.BURGERS, inputs.EULER, inputs.PERIODIC, inputs.TRANSMISSIVE
    for P in (1, 2, 3):
        for N in (200, 211, 1000, 2500):
            for ph in (0.1, 1.3, 2.9):
                out[f"advection P{P} N{N} phase {ph}"] = (A, N, P, (0.0, 2.0), PER, lambda N=N, P=P, ph=ph: _sine(N, P, 0.75, ph),
                                                          ("until", 2.0 if N <= 1000 else 0.2), {})
    for P in range(1, 7):
        if P > 3:
            out[f"advection P{P}"] = (A, 300, P, (0.0, 2.0), PER, lambda P=P: _sine(300, P, 0.75, 0.4), ("step", 101), {})
        for N in (200, 2100):
            out[f"burgers P{P} N{N}"] = (B, N, P, (0.0, 2.0), PER, lambda N=N, P=P: _sine(N, P, 0.25, 0.7, 0.5), ("step", 61), {})
            for bc in (PER, TR):
                out[f"wave P{P} N{N} bc{bc}"] = (E, N, P, (0.0, 1.0), bc, lambda N=N, P=P, bc=bc: _wave(N, P, 0.7, bc), ("step", 41), {})
            out[f"tube P{P} N{N}"] = (E, N, P, (0.0, 1.0), TR, lambda N=N, P=P: _tube(N, P), ("step", 33), {})
            out[f"tube P{P} N{N} until"] = (E, N, P, (0.0, 1.0), TR, lambda N=N, P=P: _tube(N, P), ("until", 0.05), {})
        for alpha in (1.0, 3.0):
            out[f"tube P{P} alpha {alpha}"] = (E, 500, P, (0.0, 1.0), TR, lambda P=P: _tube(500, P), ("step", 21), {"alpha": alpha})
            out[f"burgers P{P} alpha {alpha}"] = (B, 500, P, (0.0, 2.0), PER, lambda P=P: _sine(500, P, 0.25, 0.7, 0.5),
                                                  ("step", 21), {"alpha": alpha})
        out[f"wave P{P} no limiter"] = (E, 500, P, (0.0, 1.0), TR, lambda P=P: _wave(500, P, 0.2, TR), ("step", 21), {"limiter": False})
        out[f"wave P{P} eps 1e-6"] = (E, 500, P, (0.0, 1.0), TR, lambda P=P: _wave(500, P, 0.2, TR), ("step", 21), {"eps": 1e-6})
    out["wave P1 eps 1e-2 alpha 3"] = (E, 500, 1, (0.0, 1.0), TR, lambda: _wave(500, 1, 0.2, TR), ("step", 21), {"eps": 1e-2, "alpha": 3.0})
    return out


def mixed_marches():
    out = {}
    B, E, PER, TR, A = inputs.BURGERS, inputs.EULER, inputs.PERIODIC, inputs.TRANSMISSIVE, inputs.ADVECTION
    for P in range(1, 7):
        for N in (200, 3000, 5000):
            for tb in (1, 2):
                o = {"precision": wcc.FP32_MIXED, "tb_depth": tb}
                out[f"wave P{P} N{N} depth {tb}"] = (E, N, P, (0.0, 1.0), PER, lambda N=N, P=P: _wave(N, P, 0.7, PER), ("step", 60), o)
                out[f"tube P{P} N{N} depth {tb}"] = (E, N, P, (0.0, 1.0), TR, lambda N=N, P=P: _tube(N, P), ("step", 30), o)
            o = {"precision": wcc.FP32_MIXED}
            out[f"burgers P{P} N{N}"] = (B, N, P, (0.0, 2.0), PER, lambda N=N, P=P: _sine(N, P, 0.25, 0.7, 0.5), ("step", 60), o)
            out[f"advection P{P} N{N}"] = (A, N, P, (0.0, 2.0), PER, lambda N=N, P=P: _sine(N, P, 0.25, 0.7, 0.5), ("step", 60), o)
    return out


class _Member:
    def __init__(self, N, P, bc, q):
        self.system, self.N, self.P, self.x_l, self.x_r, self.bc, self.q0 = inputs.EULER, N, P, 0.0, 1.0, bc, q


def batch_digest():
    members = [_Member(N, P, inputs.TRANSMISSIVE, _tube(N, P)) if N % 2 else _Member(N, P, inputs.PERIODIC, _wave(N, P, 0.7, inputs.PERIODIC))
               for N, P in ((200, 2), (301, 3), (777, 2), (1500, 3), (2601, 3))]
    with wcc.Batch(members) as b:
        b.set_initial([m.q0 for m in members])
        b.step(30, CFL[3])
        h = hashlib.sha256()
        for i, q in enumerate(b.get_dofs()):
            h.update((np.ascontiguousarray(q) + 0.0).tobytes())
            h.update(np.ascontiguousarray(b.dt_history(i)).tobytes())
    return h.hexdigest()


def digest(march):
    system, N, P, domain, bc, data, how, options = march
    with wcc.Solver(system, N, P, domain, bc, **options) as s:
        s.set_initial(data())
        if how[0] == "until":
            s.step_until(how[1], CFL[P])
        else:
            s.step(how[1], CFL[P])
        q, dts = s.get_dofs(), s.dt_history()
    return hashlib.sha256((np.ascontiguousarray(q) + 0.0).tobytes() + np.ascontiguousarray(dts).tobytes()).hexdigest()


def _recorded(name):
    with open(os.path.join(GOLDEN, name)) as f:
        return dict(line.rstrip("\n").rsplit("  ", 1) for line in f if line.strip())


@pytest.mark.parametrize("name", list(marches()))
def test_same_bits(name):
    assert digest(marches()[name]) == _recorded("fp64_marches_1d.txt")[name]


@pytest.mark.parametrize("name", list(mixed_marches()))
def test_same_bits_mixed(name):
    assert digest(mixed_marches()[name]) == _recorded("mixed_marches_1d.txt")[name]


def test_same_bits_batch():
    assert batch_digest() == _recorded("mixed_marches_1d.txt")["batch"]
