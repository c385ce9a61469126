"""The network input formed inside the stage's line kernel (a warp's lanes exchange what neighbouring cells
share) equals that of the image kernel (a thread forms a face alone), bit for bit: js_step_vjp keeps the network
input and activations of its own forward stages, which run the line kernel; the reverse of a taped step forms
them again with the image kernel.  Every adjoint and the weight gradient depend on each pixel."""
import numpy as np
import pytest

import oracle as O
from paper_2601_04400_gb300 import workloads as W
from jsutil import to_dev

pytestmark = pytest.mark.gpu


def _state(prob, seed, jump):
    rng = np.random.default_rng(seed)
    Wp = W.random_state(prob, seed=seed, amp=0.05)
    if jump:  # density and pressure jumps, velocities at rest beside them (small values of every size)
        high = rng.random((prob.ny, prob.nx)) < 0.2
        Wp[1:3] = 10.0 ** rng.uniform(-14, -1, (2, prob.ny, prob.nx)) * rng.standard_normal((2, prob.ny, prob.nx))
        Wp[0][high] *= 20.0
        Wp[3][high] *= 20.0
        Wp[1][high] += 0.5
    return O.prim_to_cons(prob, Wp)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("jump", [False, True])
@pytest.mark.parametrize("case", ["riemann_70x45", "body_70x45", "periodic_29x57", "periodic_300x200"])
def test_images_of_line_kernel_and_image_kernel_agree(case, jump, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04400_gb300 import binding as B
    from paper_2601_04400_gb300 import neural as NN
    if case == "riemann_70x45":
        p = W.riemann2d(70, ny=45)
    elif case == "body_70x45":
        p = W.shock_cylinder(nx=70, ny=45, Lx=3.5, Ly=2.25, centre=(1.6, 1.1), radius=0.45, x_shock=0.8, viscous=True)
    else:
        nx, ny = (29, 57) if case == "periodic_29x57" else (300, 200)
        p = W.random_periodic(nx, ny, seed=1, mu=1e-3)
    U = to_dev(_state(p, 3, jump))
    s = B.Solver.from_problem(p)
    dt = 0.2 * s.max_dt(U, 0.3)
    wb = torch.zeros(B.JS_NN_NPARAM, dtype=torch.float64, device="cuda")
    s.set_neural(NN.init_weights(0, zero_last=False) * 0.5, NN.frame_norm(U, scale=0.02), w_bar=wb, precision=prec)
    lam = torch.randn(U.shape, generator=torch.Generator().manual_seed(2), dtype=torch.float64).cuda()
    pa, pb = (torch.zeros(B.JS_NPARAM, dtype=torch.float64, device="cuda") for _ in range(2))
    la, _ = s.step_vjp(U, dt, lam, None, pa)
    wa = wb.clone()
    wb.zero_()
    s.tape_reserve(1)
    s.step_taped(U.clone(), dt, 0)
    lt, _ = s.step_vjp_taped(0, dt, lam, None, pb)
    assert torch.isfinite(la).all() and float(wa.abs().max()) > 0
    assert torch.equal(la, lt)
    assert torch.equal(pa, pb)
    assert torch.equal(wa, wb)
    s.close()
