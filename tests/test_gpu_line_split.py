"""The stage kernel whose four warps share a line (grids of up to 160 blocks of eight lines) equals the
one-warp-a-line kernel bit for bit: lines and chunks of 28 cells with every remainder that matters, the
grids on both sides of the rule, a body, data that takes the first-order fallback and the FP64
reconstruction (jumps of more than 16)."""
import numpy as np
import pytest

import oracle as O
from paper_2601_04400_gb300 import workloads as W
from jsutil import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04400_gb300 import binding
    binding.lib()
    return binding


def _step(B, p, U, variant):
    s = B.Solver.from_problem(p)
    s.set_tuning(variant)
    Ud = to_dev(U)
    dt = 0.2 * O.max_dt(p, U, 0.5)
    s.step(Ud, dt, 2)
    dU = s.rhs(to_dev(U), to_dev(np.zeros_like(U)))
    out = to_host(Ud), to_host(dU), s.status()
    s.close()
    return out


@pytest.mark.parametrize("mu", [0.0, 2e-3])
@pytest.mark.parametrize("jump", [1.0, 60.0])
@pytest.mark.parametrize("nx,ny", [(6, 6), (7, 28), (28, 7), (29, 9), (56, 8), (57, 30), (85, 27), (128, 128), (141, 129)])
def test_shared_lines_equal_single_warp_lines(B, nx, ny, jump, mu):
    p = W.random_periodic(nx, ny, seed=nx + ny, amp=0.1, mu=mu, nu=1e-3 if mu else 0.0)
    rng = np.random.default_rng(nx)
    Wp = np.ones((4, ny, nx))
    Wp[0] = 1.0 + 0.3 * rng.random((ny, nx))
    Wp[3] = 1.0 + 0.3 * rng.random((ny, nx))
    Wp[1:3] = rng.standard_normal((2, ny, nx))
    high = rng.random((ny, nx)) < 0.3
    Wp[0][high] *= jump
    Wp[3][high] *= jump
    U = O.prim_to_cons(p, Wp)
    a, b = _step(B, p, U, 0), _step(B, p, U, 1)
    assert a[2] == b[2]
    assert a[0].tobytes() == b[0].tobytes()
    assert a[1].tobytes() == b[1].tobytes()


def test_shared_lines_with_a_body(B):
    p = W.shock_cylinder(nx=128, ny=64)
    U = O.prim_to_cons(p, p.W0)
    a, b = _step(B, p, U, 0), _step(B, p, U, 1)
    assert a[0].tobytes() == b[0].tobytes() and a[1].tobytes() == b[1].tobytes()
