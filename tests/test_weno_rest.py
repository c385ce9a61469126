"""Velocities near rest beside a jump: a face state there is far below the stencil's largest difference, so
the integer reconstruction (csrc/js_weno.cuh) takes each candidate on its own scale (weno_fits).  On the CPU: face states as accurate as the FP64 sequence's, ordinary velocity fields on
the one common scale.  On the GPU: fluxes and gradients of gas near rest.

Tolerances.  u = 2^-53.  The FP64 sequence rounds a difference (1), a candidate (2), an indicator (5, squared
and multiplied with another's in a weight: 22 with its products) and the quotient (3): its error is below
28 u S with S = |q| + the weighted sum of the candidates' absolute terms; the integer form is held to 16 u S.
A tangential momentum flux is the mass flux (10 u) times a face state (16 u S, S below 2 |v|): 64 u |v|
times the mass flux covers the two faces of a cell.  A derivative of a face state sums terms below 43 (34
from the weights, 9 from the candidates) of 16 u each: 700 u, and a Jacobian entry a few of them."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle as O
from paper_2601_04400_gb300 import workloads as W

SRC = r"""
#include <cstdio>
#include "js_weno.cuh"
using namespace js;
int main() {
  double v[5];
  while (std::fread(v, 8, 5, stdin) == 5) {
    const Qx m2 = qx_of(v[0]), m1 = qx_of(v[1]), x = qx_of(v[2]), p1 = qx_of(v[3]), p2 = qx_of(v[4]);
    const Fx a = fx_of(m1, m2), b = fx_of(x, m1), c = fx_of(p1, x), d = fx_of(p2, p1);
    const int EL = imax(a.e, b.e), EM = imax(b.e, c.e), ER = imax(c.e, d.e), F = imax(EL, ER);
    Sm s0, s1, s2, t, u;
    sm_pair(a, b, t, s0, u);
    sm_pair(c, d, t, u, s2);
    sm_pair(b, c, s1, t, u);
    double o[3];
    o[2] = weno_fits(x, EL, EM, ER, F) ? 1.0 : 0.0;
    weno_faces(x, a, b, c, d, s0, s1, s2, F, o[0], o[1], o[2] > 0);
    std::fwrite(o, 8, 3, stdout);
  }
  return 0;
}
"""
U = 2.0 ** -53
LD = np.longdouble


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("weno_rest")
    (d / "t.cpp").write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_04400_gb300", "csrc")
    subprocess.run([gxx, "-O2", "-std=gnu++17", "-I", inc, str(d / "t.cpp"), "-o", str(d / "t")], check=True)

    def f(q):
        r = subprocess.run([str(d / "t")], input=np.ascontiguousarray(q).tobytes(), stdout=subprocess.PIPE, check=True)
        o = np.frombuffer(r.stdout).reshape(-1, 3)
        return o[:, :2], o[:, 2] > 0
    return f


def _faces(q):
    """Face states in extended precision and the scale S of each."""
    q = q.astype(LD)
    a, b, c, d = (q[:, k + 1] - q[:, k] for k in range(4))
    eps = LD(1) / LD(10 ** 6)
    beta = [LD(13) / 12 * D ** 2 + t ** 2 / 4 + eps for D, t in ((b - a, 3 * b - a), (c - b, b + c), (d - c, d - 3 * c))]
    faces, scales = [], []
    for lin, e in (((1, 6, 3), [(-2, 5, 0, 0), (0, 1, 2, 0), (0, 0, 4, -1)]),
                   ((3, 6, 1), [(1, -4, 0, 0), (0, -2, -1, 0), (0, 0, -5, 2)])):
        w = [lin[k] / beta[k] ** 2 for k in range(3)]
        s = w[0] + w[1] + w[2]
        terms = [[w[k] / s * e[k][j] * x / 6 for j, x in enumerate((a, b, c, d))] for k in range(3)]
        faces.append(q[:, 2] + sum(t for r in terms for t in r))
        scales.append(abs(q[:, 2]) + sum(abs(t) for r in terms for t in r))
    return np.stack(faces, axis=1), np.stack(scales, axis=1)


N = 40000


def _near_rest(rng):
    v = 10.0 ** rng.uniform(-14, 0, (N, 1)) * rng.standard_normal((N, 5)) * (rng.random((N, 1)) < 0.9)
    side = (np.arange(5) < rng.integers(1, 5, (N, 1))) ^ (rng.random((N, 1)) < 0.5)
    J = 10.0 ** rng.uniform(-4, 4, (N, 1))
    return v * J + side * J * (1 + 0.01 * rng.random((N, 5)))


def _noise(rng):
    return 10.0 ** rng.uniform(-6, 3, (N, 1)) * rng.standard_normal((N, 5))


def _crossing(rng):
    h = 10.0 ** rng.uniform(-3, -0.3, (N, 1))
    return 10.0 ** rng.uniform(-6, 3, (N, 1)) * np.sin(h * (np.arange(5) - 2 + 0.1 * rng.standard_normal((N, 1))))


def _scattered(rng):
    d = 10.0 ** rng.uniform(-9, 1, (N, 5)) * rng.choice([-1.0, 1.0], (N, 5))
    return np.cumsum(d, axis=1) - d[:, :1] * (rng.random((N, 1)) < 0.5)


@pytest.mark.parametrize("field,most", [(_near_rest, 1.0), (_noise, 0.005), (_crossing, 0.001), (_scattered, 1.0)])
def test_integer_faces_of_velocities(run, field, most):
    """`most`: the share of cells that may leave the common scale."""
    q = field(np.random.default_rng(3))
    o, fits = run(q)
    want, scale = _faces(q)
    assert np.mean(~fits) <= most
    assert float(np.max(np.abs(o - want) / np.where(scale > 0, scale, 1))) <= 16 * U


def _tube(n, J, quiet, u, p):
    """A 1D row: tangential velocity J on the left half, `quiet` small values on the right."""
    prob = W.sod(n)
    Wp = np.ones((4, 1, n))
    Wp[1], Wp[3] = u, p
    Wp[2, 0] = np.where(np.arange(n) < n // 2, J, quiet * (1 + 0.3 * np.sin(np.arange(n))))
    return prob, O.prim_to_cons(prob, Wp)


def _solver(prob):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04400_gb300 import binding as B
    return B.Solver.from_problem(prob)


@pytest.mark.gpu
@pytest.mark.parametrize("quiet", [1e-6, 1e-9, 1e-12])
def test_momentum_of_gas_near_rest(quiet):
    """The flow goes left, so the quiet side is upwind: its momentum rate is of the order of its velocity."""
    from jsutil import to_dev, to_host
    n = 64
    prob, U0 = _tube(n, 1.0, quiet, -0.5, 1.0)
    s = _solver(prob)
    got = to_host(s.rhs(to_dev(U0)))[2, 0]
    want = O.rhs(prob, U0)[2, 0]
    s.close()
    cells = slice(n // 2, n)
    assert np.max(np.abs(want[cells])) < 10 * quiet / prob.dx
    assert np.max(np.abs(got - want)[cells]) <= 2 * 64 * U * (1.3 * quiet) * 0.5 / prob.dx  # (both sides' rounding)


@pytest.mark.gpu
@pytest.mark.parametrize("J,quiet", [(1e3, 1e-3), (1e3, 1e-6), (30.0, 1e-3)])
def test_gradient_of_gas_near_rest(J, quiet):
    """Rows of the Jacobian d(rho v)'_c / d(rho v)_k at the cells c beside the jump."""
    from jsutil import to_dev, to_host
    n = 32
    prob, U0 = _tube(n, J, quiet, -500.0, 1e6)
    s = _solver(prob)
    cols = []
    for k in range(n):
        dU = np.zeros_like(U0)
        dU[2, 0, k] = 1.0
        cols.append(O.rhs_tangent(prob, U0, dU, np.zeros(20))[1][2, 0])
    want = np.stack(cols, axis=1)  # [c][k]
    for c in range(n // 2 - 1, n // 2 + 3):
        lam = np.zeros_like(U0)
        lam[2, 0, c] = 1.0
        got = to_host(s.rhs_vjp(to_dev(U0), to_dev(lam))[0])[2, 0]
        assert np.max(np.abs(got - want[c])) <= 1000 * U * np.max(np.abs(want[c]))
    s.close()
