"""The reverse line kernel whose four warps share a line (small grids, js_step_vjp) against the one whose
warps take a line each (js_batch_step_vjp): the same device functions compiled twice, so lambda and the
parameter gradient agree to rounding (other products may be contracted), over line and chunk remainders,
with first-order fallback faces and jumps that take the FP64 reconstruction."""
import numpy as np
import pytest

import oracle as O
from paper_2601_04400_gb300 import workloads as W
from jsutil import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mu", [0.0, 2e-3])
@pytest.mark.parametrize("jump", [1.0, 60.0])
@pytest.mark.parametrize("nx,ny", [(6, 6), (26, 9), (27, 7), (54, 8), (55, 31), (83, 26), (128, 128), (141, 129)])
def test_shared_lines_equal_single_warp_lines(nx, ny, jump, mu):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04400_gb300 import binding as B
    p = W.random_periodic(nx, ny, seed=nx + ny, amp=0.1, mu=mu, nu=1e-3 if mu else 0.0)
    rng = np.random.default_rng(nx)
    Wp = np.ones((4, ny, nx))
    Wp[0] = 1.0 + 0.3 * rng.random((ny, nx))
    Wp[3] = 1.0 + 0.3 * rng.random((ny, nx))
    Wp[1:3] = 0.3 * rng.standard_normal((2, ny, nx))
    high = rng.random((ny, nx)) < 0.2
    Wp[0][high] *= jump
    Wp[3][high] *= jump
    U = O.prim_to_cons(p, Wp)
    dt = 0.1 * O.max_dt(p, U, 0.5)
    lam = rng.standard_normal(U.shape)
    s = B.Solver.from_problem(p)
    pa = torch.zeros(20, dtype=torch.float64, device="cuda")
    la, _ = s.step_vjp(to_dev(U), dt, to_dev(lam), None, pa)
    s.close()
    b = B.Batch([p])
    Ud, out = to_dev(U), to_dev(np.zeros_like(U))
    pb = torch.zeros(20, dtype=torch.float64, device="cuda")
    b.set_states([Ud.clone()])
    b.step_vjp([Ud], [dt], [to_dev(lam)], [out], [pb])
    assert b.status() == 0
    b.close()
    a, c = to_host(la), to_host(out)
    assert np.all(np.isfinite(a))
    assert np.max(np.abs(a - c)) <= 1e-12 * np.max(np.abs(c))
    assert float((pa - pb).abs().max()) <= 1e-11 * float(pb.abs().max())
