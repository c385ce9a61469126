"""Velocities near and below the normal range (a front's decay into gas at rest passes through them), against
the oracle: the integer reconstruction takes subnormal values and gives subnormal results.

Tolerance: u = 2^-53.  A tangential momentum flux is the mass flux (10 u) times a face state (28 u of
|v| and the candidates, below 3 |v|): below 100 u |v| for the two faces of a cell and the division by dx, plus
one unit of the subnormal range, 2^-1074, for each of some 30 roundings (times the mass flux over dx)."""
import numpy as np
import pytest

import oracle as O
from paper_2601_04400_gb300 import workloads as W
from jsutil import to_dev, to_host

pytestmark = pytest.mark.gpu


def _rates(prob, v, axis):
    """d(momentum of the tangential velocity v)/dt of a uniform flow along `axis`, from both sides."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04400_gb300 import binding as B
    Wp = np.ones((4, prob.ny, prob.nx))
    Wp[1 + axis] = -0.5
    Wp[2 - axis] = v if axis == 0 else v.T
    U0 = O.prim_to_cons(prob, Wp)
    s = B.Solver.from_problem(prob)
    got = to_host(s.rhs(to_dev(U0)))[2 - axis]
    assert s.status() == 0
    s.close()
    return got, O.rhs(prob, U0)[2 - axis]


def _velocities(prob, kind, exponent, axis):
    n, m = (prob.nx, prob.ny) if axis == 0 else (prob.ny, prob.nx)
    i = np.arange(n)[None, :] + 0.1 * np.arange(m)[:, None]
    v = {"waves": np.sin(0.4 * i), "step": np.where(i > n / 2, 1.0, 0.0), "front": 2.0 ** (-4.0 * np.abs(i - 20))}[kind]
    return v * 2.0 ** exponent, (prob.dx if axis == 0 else prob.dy)


@pytest.mark.parametrize("exponent", [-900, -980, -1010, -1020, -1026, -1040, -1060])
@pytest.mark.parametrize("kind", ["waves", "step", "front"])
@pytest.mark.parametrize("axis", [0, 1])
def test_small_velocities(axis, kind, exponent):
    prob = W.random_periodic(60, 40, seed=1)
    v, h = _velocities(prob, kind, exponent, axis)
    got, want = _rates(prob, v, axis)
    assert np.any(want)
    tol = 100 * 2.0 ** -53 * np.max(np.abs(v)) + 30 * 2.0 ** -1074
    assert np.max(np.abs(got - want)) <= 2 * tol * 0.5 / h
