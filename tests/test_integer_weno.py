"""The integer arithmetic of the fast kernels (csrc/js_wide.cuh, csrc/js_weno.cuh), compiled for the host,
against extended precision: reciprocals, reciprocal square roots and sound speeds, WENO5 face states and
the derivatives of a face's correction with respect to the cell's four differences.

Tolerances: a wide routine rounds a value of at least 56 correct bits once, so its relative error is
below 2^-53 + 2^-56.  A face state adds to its rounding about 2^-57 of the largest difference per
fixed-point operation, some tens of them: 2^-53 |q| + 2^-52 max |d|.  A derivative (below 16) sums about
thirty terms held to 2^-56 of values below 16: 2^-47."""
import os
import shutil
import subprocess

import numpy as np
import pytest

SRC = r"""
#include <cstdio>
#include <vector>
#include "js_weno.cuh"
using namespace js;
int main(int argc, char** argv) {
  const bool wide = argv[1][0] == 'w';
  const int ni = wide ? 3 : 5, no = wide ? 3 : 10;
  std::vector<double> in, out;
  double v[5];
  while (std::fread(v, 8, ni, stdin) == (size_t)ni) {
    double o[10];
    if (wide) {
      o[0] = recip_wide(v[0]);
      o[1] = rsqrt_wide(v[0]);
      o[2] = sound_wide(v[0], v[1], v[2]);
    } else {
      const Qx m2 = qx_of(v[0]), m1 = qx_of(v[1]), x = qx_of(v[2]), p1 = qx_of(v[3]), p2 = qx_of(v[4]);
      const Fx a = fx_of(m1, m2), b = fx_of(x, m1), c = fx_of(p1, x), d = fx_of(p2, p1);
      const int F = imax(imax(a.e, b.e), imax(c.e, d.e));
      Sm s0, s1, s2, t, u;
      Lv v0, v1, v2, y, z;
      sm_pair_grad(a, b, t, s0, u, y, v0, z);
      sm_pair_grad(c, d, t, u, s2, y, z, v2);
      sm_pair_grad(b, c, s1, t, u, v1, y, z);
      weno_faces(x, a, b, c, d, s0, s1, s2, F, o[0], o[1]);
      const GradCell g = grad_cell(a, b, c, d, s0, s1, s2, v0, v1, v2, F);
      weno_grad_side(g, false, o + 2);
      weno_grad_side(g, true, o + 6);
    }
    std::fwrite(o, 8, no, stdout);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("integer_weno")
    (d / "t.cpp").write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_04400_gb300", "csrc")
    subprocess.run([gxx, "-O2", "-std=gnu++17", "-I", inc, str(d / "t.cpp"), "-o", str(d / "t")], check=True)

    def f(mode, x, n):
        r = subprocess.run([str(d / "t"), mode], input=np.ascontiguousarray(x).tobytes(), stdout=subprocess.PIPE, check=True)
        return np.frombuffer(r.stdout).reshape(-1, n)
    return f


LD = np.longdouble


@pytest.mark.parametrize("scale", [1.0, 1e-90, 1e90])
def test_wide_reciprocals_and_sound_speeds(run, scale):
    rng = np.random.default_rng(1)
    x = np.exp(rng.uniform(-6, 6, (20000, 3))) * scale
    x[:64, 0] = scale * 2.0 ** np.arange(-32, 32)  # powers of two
    x[64:128, 0] = np.nextafter(x[:64, 0], 0)
    x[:, 1] /= scale  # (the sound speed's product stays in range)
    o = run("w", x, 3)
    e = x.astype(LD)
    want = np.stack([1 / e[:, 0], 1 / np.sqrt(e[:, 0]), np.sqrt(e[:, 0] * e[:, 1] / e[:, 2])], axis=1)
    assert float(np.max(np.abs(o - want) / want)) <= 2.0 ** -53 + 2.0 ** -56


def _exact(q):
    """Face states and d(6 (face - q))/d(a, b, c, d), left-biased then right-biased."""
    q = q.astype(LD)
    a, b, c, d = (q[:, k + 1] - q[:, k] for k in range(4))
    z = np.zeros_like(a)
    eps = LD(1) / LD(10 ** 6)
    D = [b - a, c - b, d - c]
    t = [3 * b - a, b + c, d - 3 * c]
    dD = [(-1, 1, 0, 0), (0, -1, 1, 0), (0, 0, -1, 1)]
    dt = [(-1, 3, 0, 0), (0, 1, 1, 0), (0, 0, -3, 1)]
    beta = [LD(13) / 12 * D[k] ** 2 + t[k] ** 2 / 4 + eps for k in range(3)]
    grad = [[LD(13) / 6 * D[k] * dD[k][x] + t[k] * dt[k][x] / 2 for x in range(4)] for k in range(3)]
    sides = [((1, 6, 3), [(-2, 5, 0, 0), (0, 1, 2, 0), (0, 0, 4, -1)]),
             ((3, 6, 1), [(1, -4, 0, 0), (0, -2, -1, 0), (0, 0, -5, 2)])]
    faces, ders = [], []
    for lin, e in sides:
        w = [lin[k] / beta[k] ** 2 for k in range(3)]
        s = w[0] + w[1] + w[2]
        om = [x / s for x in w]
        ek = [e[k][0] * a + e[k][1] * b + e[k][2] * c + e[k][3] * d for k in range(3)]
        C = om[0] * ek[0] + om[1] * ek[1] + om[2] * ek[2]
        faces.append(q[:, 2] + C / 6)
        ders += [sum((om[k] * e[k][x] - 2 * om[k] * (ek[k] - C) * grad[k][x] / beta[k] for k in range(3)), z)
                 for x in range(4)]
    return np.stack(faces, axis=1), np.stack(ders, axis=1)


def _stencils(kind):
    rng = np.random.default_rng(5)
    n = 20000
    if kind == "smooth":
        x = rng.uniform(0, 6, (n, 1)) + 0.05 * np.arange(5)
        return 1.5 + np.sin(x)
    if kind == "noise":
        return 1.0 + rng.random((n, 5))
    if kind == "tiny_noise":
        return 1.0 + 1e-9 * rng.standard_normal((n, 5))
    if kind == "jumps":
        return np.where(rng.random((n, 5)) < 0.5, 1.0, rng.uniform(1.0, 9.0, (n, 1)))
    if kind == "constant":
        return np.repeat(rng.uniform(0.1, 10.0, (n, 1)), 5, axis=1)
    s = {"small_scale": 1e-7, "large_scale": 1e8}[kind]
    return s * (1.0 + 0.5 * rng.random((n, 5)))


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("kind", ["smooth", "noise", "tiny_noise", "jumps", "constant", "small_scale", "large_scale"])
def test_faces_and_derivatives(run, kind, sign):
    q = sign * _stencils(kind)
    o = run("f", q, 10)
    faces, ders = _exact(q)
    dmax = np.max(np.abs(np.diff(q, axis=1)), axis=1, keepdims=True)
    err = np.abs(o[:, :2] - faces).astype(float)
    assert np.all(err <= 2.0 ** -53 * np.abs(o[:, :2]) + 2.0 ** -52 * dmax)
    assert float(np.max(np.abs(o[:, 2:] - ders))) <= 2.0 ** -47
