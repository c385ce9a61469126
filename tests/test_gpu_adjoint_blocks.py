"""Every compilation of the reverse line kernel against the oracle: grids on both sides of the block counts at
which the shared-line kernel, the kernel of three blocks an SM and the one of four take over (228 and 456 blocks
of eight lines), Euler and viscous, with remainders of lines and chunks; and batches of few and of many blocks
with viscous and inviscid instances against the per-grid calls.

Dot products: <lam, J v> (oracle, forward mode) = <J^T lam, v> (GPU) to 1e-12 of sum |lam| max |J v|, as in
test_gpu_adjoint.py.  A batched instance repeats js_step_vjp's lambda up to contraction in another compilation
(1e-12, test_gpu_adjoint_split.py)."""
import numpy as np
import pytest

import oracle as O
from paper_2601_04400_gb300 import workloads as W
from jsutil import to_dev, to_host

pytestmark = pytest.mark.gpu


def _blocks(nx, ny):
    """Blocks of eight lines of 28 cells (-1 .. n) in both directions."""
    chunks = lambda n: (n + 2 + 27) // 28  # noqa: E731
    return (ny + 7) // 8 * chunks(nx) + (nx + 7) // 8 * chunks(ny)


GRIDS = [(180, 128), (181, 129), (250, 190), (237, 189), (256, 200), (301, 203)]


def test_the_grids_lie_on_both_sides():
    n = [_blocks(*g) for g in GRIDS]
    assert n[0] <= 228 < n[1] < n[3] < n[2] <= 456 < n[4] < n[5]


def _problem(flow, nx, ny):
    if flow == "body":
        return W.shock_cylinder(nx=nx, ny=ny, Lx=6.0, Ly=6.0 * ny / nx, Re=300.0, centre=(2.0, 3.0 * ny / nx))
    if flow == "riemann":
        return W.riemann2d(nx, ny=ny)
    return W.random_periodic(nx, ny, seed=2, mu=2e-3, nu=1e-3)


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04400_gb300 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("flow", ["riemann", "body", "periodic"])
@pytest.mark.parametrize("nx,ny", GRIDS)
def test_step_vjp_dot_product(B, nx, ny, flow):
    prob = _problem(flow, nx, ny)
    U = O.prim_to_cons(prob, W.random_state(prob, seed=7, amp=0.02))
    dt = 0.4 * O.max_dt(prob, U, 0.5)
    rng = np.random.default_rng(3)
    v = rng.standard_normal(U.shape) * np.abs(U).max(axis=(1, 2), keepdims=True) * 1e-3
    dth = np.zeros(20)
    dth[0] = 0.1
    if prob.mu > 0:
        dth[1] = 1e-3
    if prob.nu > 0:
        dth[3] = 1e-3
    lam = rng.standard_normal(U.shape)
    _, Jv = O.step_tangent(prob, U, v, dth, [dt])
    s = B.Solver.from_problem(prob)
    Ub, pb = s.step_vjp(to_dev(U), dt, to_dev(lam))
    assert s.status() == 0
    s.close()
    lhs = np.dot(lam.reshape(-1), Jv.reshape(-1))
    rhs = np.dot(to_host(Ub).reshape(-1), v.reshape(-1)) + np.dot(to_host(pb), dth)
    assert abs(lhs - rhs) <= 1e-12 * np.abs(lam).sum() * np.abs(Jv).max()


@pytest.mark.parametrize("flows", [("riemann", "body"), ("riemann",), ("periodic",)])
@pytest.mark.parametrize("many", [False, True])
def test_batched_reverse_equals_step_vjp(B, many, flows):
    import torch
    sizes = [(181, 129), (250, 190), (141, 97)] if many else [(90, 70), (70, 90)]
    probs = [_problem(flows[k % len(flows)], nx, ny) for k, (nx, ny) in enumerate(sizes + sizes[:1])]
    total = sum(_blocks(p.nx, p.ny) for p in probs)
    assert (total > 456) == many
    rng = np.random.default_rng(5)
    U = [to_dev(O.prim_to_cons(p, W.random_state(p, seed=k, amp=0.02))) for k, p in enumerate(probs)]
    lam = [to_dev(rng.standard_normal(tuple(u.shape))) for u in U]
    dts, ref = [], []
    for p, u, l in zip(probs, U, lam):
        s = B.Solver.from_problem(p)
        dts.append(0.4 * s.max_dt(u, 0.5))
        ref.append(tuple(x.clone() for x in s.step_vjp(u, dts[-1], l)))
        s.close()
    b = B.Batch(probs)
    b.set_states([u.clone() for u in U])
    out = [torch.empty_like(u) for u in U]
    pb = [torch.zeros(B.JS_NPARAM, dtype=torch.float64, device="cuda") for _ in U]
    b.step_vjp(U, dts, lam, out, pb)
    assert b.status() == 0
    b.close()
    for o, g, (l, p) in zip(out, pb, ref):
        assert float((o - l).abs().max()) <= 1e-12 * float(l.abs().max())
        assert float((g - p).abs().max()) <= 1e-11 * float(p.abs().max())
