"""The reverse pass is linear in the adjoint it is given, down to the subnormal range: adjoints of 2^-1040
times a reference's give 2^-1040 times its result, up to the rounding of subnormal numbers.

Tolerance: a result passes a few hundred roundings of 2^-1074, each multiplied on by at most some 10
(derivatives of the flux and the reconstruction) and 1/dx twice (differences, then viscous terms): 1e3 x 10 x
64^2 units of 2^-1074, 2e-3 of the smallest step 2^-1040 1/dx that a lost term would make."""
import numpy as np
import pytest

import oracle as O
from paper_2601_04400_gb300 import workloads as W
from jsutil import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mu", [0.0, 2e-3])
@pytest.mark.parametrize("nx,ny", [(64, 1), (60, 40), (260, 200)])
def test_reverse_of_tiny_adjoints(nx, ny, mu):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04400_gb300 import binding as B
    if ny == 1:
        prob = W.sod(nx).with_(mu=mu)
        U = O.prim_to_cons(prob, W.random_state(prob, seed=3, amp=0.2))
    else:
        prob = W.random_periodic(nx, ny, seed=3, mu=mu).with_(dx=1 / 64, dy=1 / 64)
        U = O.prim_to_cons(prob, W.random_state(prob, seed=3, amp=0.2))
    lam = np.random.default_rng(5).standard_normal(U.shape)
    s = B.Solver.from_problem(prob)
    Ud = to_dev(U)
    want = to_host(s.rhs_vjp(Ud, to_dev(lam))[0])
    got = to_host(s.rhs_vjp(Ud, to_dev(lam * 2.0 ** -1040))[0])
    assert s.status() == 0
    s.close()
    err = np.abs(got * 2.0 ** 520 * 2.0 ** 520 - want)
    assert np.max(err) <= 1e3 * 10 * 64 ** 2 * 2.0 ** -34
