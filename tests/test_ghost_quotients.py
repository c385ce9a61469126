"""Quotients of the immersed-boundary ghost fill (velocities of the source cells, internal energy): within
0.53 ulp, as near as IEEE division but for one in a few dozen (csrc/js_wide.cuh: quot_wide, compiled for the
host; js_fill.cuh: ib_image on the GPU).

Tolerances.  The quotient is held to 57 bits and rounded once: 2^-53 + 2^-57.  Its error before rounding,
below 2^-4 ulp, moves at most one in eight results to the other neighbour, and a product with it (the ghost's
momentum) no more; a reciprocal multiplied (up to 1.5 ulp) misses one in four."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle as O
from paper_2601_04400_gb300 import workloads as W

SRC = r"""
#include <cstdio>
#include "js_wide.cuh"
int main() {
  double v[2];
  while (std::fread(v, 8, 2, stdin) == 2) {
    const double q = js::quot_wide(v[0], v[1], js::recip_top(js::mant64(v[1])));
    std::fwrite(&q, 8, 1, stdout);
  }
  return 0;
}
"""


def _quotients(tmp_path, x):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    (tmp_path / "t.cpp").write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_04400_gb300", "csrc")
    subprocess.run([gxx, "-O2", "-std=gnu++17", "-I", inc, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t")], check=True)
    r = subprocess.run([str(tmp_path / "t")], input=np.ascontiguousarray(x).tobytes(), stdout=subprocess.PIPE, check=True)
    return np.frombuffer(r.stdout)


@pytest.mark.parametrize("scale", [(1.0, 1.0), (1e-150, 1e150), (1e150, 1e-150), (1e-295, 1e-5), (1e290, 1e295)])
def test_wide_quotients(tmp_path, scale):
    rng = np.random.default_rng(4)
    x = np.exp(rng.uniform(-5, 5, (40000, 2))) * rng.choice([-1.0, 1.0], (40000, 2))
    x[:40, 0] = 2.0 ** np.arange(-20, 20)  # powers of two and their neighbours
    x[40:80, 1] = 2.0 ** np.arange(-20, 20)
    x[80:120] = np.nextafter(x[:40], 0)
    x[120:160, 0] = x[120:160, 1]
    x[160, 0] = 0.0
    x *= np.array(scale)
    q = _quotients(tmp_path, x)
    want = x[:, 0].astype(np.longdouble) / x[:, 1].astype(np.longdouble)
    assert q[160] == 0.0
    ok = want != 0
    assert float(np.max(np.abs(q - want)[ok] / np.abs(want)[ok])) <= 2.0 ** -53 + 2.0 ** -57
    assert np.mean(q == x[:, 0] / x[:, 1]) >= 7 / 8


@pytest.mark.gpu
def test_ghost_momenta_of_a_flat_wall():
    """A wall along a cell face on a binary grid: every image point is a cell centre, so a ghost's momentum is
    the density times the rounded quotient of its one source cell.  A step of vanishing size leaves the
    fluid as it is and the ghosts filled."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04400_gb300 import binding as B
    from jsutil import to_dev, to_host
    nx, ny, jw = 256, 32, 12
    h = 1.0 / 64
    y = (np.arange(ny) + 0.5) * h
    sdf = np.repeat((y - jw * h)[:, None], nx, axis=1)
    prob = W.random_periodic(nx, ny, seed=2).with_(dx=h, dy=h, x0=0.0, y0=0.0, sdf=sdf, bc=(2, 2, 0, 0))
    rng = np.random.default_rng(8)
    Wp = np.empty((4, ny, nx))
    Wp[0] = rng.uniform(0.5, 2.0, (ny, nx))
    Wp[1:3] = rng.standard_normal((2, ny, nx))
    Wp[3] = rng.uniform(0.5, 2.0, (ny, nx))
    U0 = O.prim_to_cons(prob, Wp)
    U0[1:3] = rng.uniform(-1, 1, (2, ny, nx))
    U0[3] += 5.0
    s = B.Solver.from_problem(prob)
    U = to_host(s.step(to_dev(U0), 1e-300, 1))
    assert s.status() == 0
    s.close()
    for k in range(3):
        src, g = jw + k, jw - 1 - k
        assert np.array_equal(U[0, g], U0[0, src])
        for c, sign in ((1, 1.0), (2, -1.0)):
            assert np.mean(U[c, g] == sign * U0[0, src] * (U0[c, src] / U0[0, src])) >= 7 / 8
