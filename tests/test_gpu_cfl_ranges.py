"""The step size of js_max_dt and js_step_cfl bit for bit against the oracle's around the limits of
the reduction's approximations: the grid size from which it takes two passes, the energy ratio and
the magnitudes up to which pass 1 uses FP32, and rates that differ by less than its margin."""
import numpy as np
import pytest

import oracle as O
from paper_2601_04400_gb300 import workloads as W
from jsutil import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04400_gb300 import binding
    binding.lib()
    return binding


def _check(B, p, U):
    import torch
    s = B.Solver.from_problem(p)
    Ud = to_dev(U)
    want = O.max_dt(p, U, 0.5)
    assert s.max_dt(Ud, 0.5) == want
    log = torch.zeros(1, dtype=torch.float64, device="cuda")
    s.step_cfl(Ud, 0.5, 1, dt_log=log)
    assert log.item() == want
    s.close()


@pytest.mark.parametrize("mu", [0.0, 2e-3])
@pytest.mark.parametrize("nx,ny", [(181, 181), (182, 181), (517, 301), (32768, 1), (33000, 1)])
@pytest.mark.parametrize("scale", ["one", "tiny", "large"])
@pytest.mark.parametrize("e_over_p", [3.0, 38.0, 42.0, 1e7])
def test_step_size_equals_the_oracles(B, nx, ny, mu, scale, e_over_p):
    """gamma - 1 = 0.4: internal over total energy is 1/16 at E/p = 40.  The scales put density and
    energy inside and outside the FP32 range."""
    base = W.sod(nx) if ny == 1 else W.riemann2d(nx, ny=ny)
    p = base.with_(mu=mu if scale == "one" else 0.0)
    rng = np.random.default_rng(nx + ny)
    Wp = 1.0 + 0.1 * rng.standard_normal((4, ny, nx))
    Wp[1:3] -= 1.0
    if ny == 1:
        Wp[2] = 0.0
    j, i = ny // 2, min(nx - 1, 255)
    press = 1.3
    u = np.sqrt(2.0 * press * (e_over_p - 1.0 / 0.4))
    Wp[:, j, i] = (1.0, u, 0.0, press)
    d = {"one": 1.0, "tiny": 1e-14, "large": 1e14}[scale]
    Wp[0] *= d
    Wp[3] *= d
    _check(B, p, O.prim_to_cons(p, Wp))


@pytest.mark.parametrize("spread", [1e-13, 1e-6, 1e-5, 1e-4])
def test_rates_within_the_margin(B, spread):
    p = W.riemann2d(300, ny=300)
    rng = np.random.default_rng(7)
    Wp = np.ones((4, 300, 300))
    Wp[1] = 2.0 * (1.0 + spread * rng.standard_normal((300, 300)))
    Wp[2] = -0.7
    _check(B, p, O.prim_to_cons(p, Wp))
