"""Small derivatives of a face state: beside a jump the far stencils' weights are 1e-12 and less, and so are
the derivatives with respect to their differences.  They are formed on the scale of their own weights
(csrc/js_weno.cuh: weno_grad_side), compiled for the host here, and compared with extended precision.

Tolerance: u = 2^-53.  A derivative sums products of a weight, a candidate difference and an indicator's
logarithmic derivative.  In FP64 these carry 22, 3 and 8 roundings and the product 2: below 35 u of the sum
of the terms' magnitudes to first order; the integer form is held to 32 u of that sum."""
import os
import shutil
import subprocess

import numpy as np
import pytest

SRC = r"""
#include <cstdio>
#include "js_weno.cuh"
using namespace js;
int main() {
  double v[5];
  while (std::fread(v, 8, 5, stdin) == 5) {
    const Qx m2 = qx_of(v[0]), m1 = qx_of(v[1]), x = qx_of(v[2]), p1 = qx_of(v[3]), p2 = qx_of(v[4]);
    const Fx a = fx_of(m1, m2), b = fx_of(x, m1), c = fx_of(p1, x), d = fx_of(p2, p1);
    const int F = imax(imax(a.e, b.e), imax(c.e, d.e));
    Sm s0, s1, s2, t, u;
    Lv v0, v1, v2, y, z;
    sm_pair_grad(a, b, t, s0, u, y, v0, z);
    sm_pair_grad(c, d, t, u, s2, y, z, v2);
    sm_pair_grad(b, c, s1, t, u, v1, y, z);
    const GradCell g = grad_cell(a, b, c, d, s0, s1, s2, v0, v1, v2, F);
    double o[8];
    weno_grad_side(g, false, o);
    weno_grad_side(g, true, o + 4);
    std::fwrite(o, 8, 8, stdout);
  }
  return 0;
}
"""
U = 2.0 ** -53
LD = np.longdouble
N = 20000


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("weno_derivative")
    (d / "t.cpp").write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_04400_gb300", "csrc")
    subprocess.run([gxx, "-O2", "-std=gnu++17", "-I", inc, str(d / "t.cpp"), "-o", str(d / "t")], check=True)

    def f(q):
        r = subprocess.run([str(d / "t")], input=np.ascontiguousarray(q).tobytes(), stdout=subprocess.PIPE, check=True)
        return np.frombuffer(r.stdout).reshape(-1, 8)
    return f


def _exact(q):
    """d(6 (face - q))/d(a, b, c, d), left-biased then right-biased, and the sums of the terms' magnitudes."""
    q = q.astype(LD)
    x = [q[:, k + 1] - q[:, k] for k in range(4)]
    a, b, c, d = x
    eps = LD(12) / LD(10 ** 6)
    s = [13 * D ** 2 + 3 * t ** 2 + eps for D, t in ((b - a, 3 * b - a), (c - b, b + c), (d - c, d - 3 * c))]
    # logarithmic derivatives of the indicators, halved: coefficients of the differences
    lv = [{0: {0: 16, 1: -22}, 1: {0: -22, 1: 40}}, {1: {1: 16, 2: -10}, 2: {1: -10, 2: 16}}, {2: {2: 40, 3: -22}, 3: {2: -22, 3: 16}}]
    T = [c - 2 * b + a, d - 2 * c + b]
    Tm = [abs(c) + 2 * abs(b) + abs(a), abs(d) + 2 * abs(c) + abs(b)]
    out, mag = [], []
    for lin, de, f0, f1 in (((1, 6, 3), [(-2, 5, 0, 0), (0, 1, 2, 0), (0, 0, 4, -1)], -2, 1),
                            ((3, 6, 1), [(1, -4, 0, 0), (0, -2, -1, 0), (0, 0, -5, 2)], 1, -2)):
        w = [lin[k] / s[k] ** 2 for k in range(3)]
        tot = w[0] + w[1] + w[2]
        w = [v / tot for v in w]
        e01, e12 = f0 * T[0], f1 * T[1]
        m01, m12 = abs(f0) * Tm[0], abs(f1) * Tm[1]
        G = [w[1] * e01 + w[2] * (e01 + e12), w[2] * e12 - w[0] * e01, -w[0] * (e01 + e12) - w[1] * e12]
        Gm = [w[1] * m01 + w[2] * (m01 + m12), w[2] * m12 + w[0] * m01, w[0] * (m01 + m12) + w[1] * m12]
        for j in range(4):
            g = m = 0
            for k in range(3):
                v = sum((co * x[i] for i, co in lv[k].get(j, {}).items()), 0 * a) / s[k]
                vm = sum((abs(co * x[i]) for i, co in lv[k].get(j, {}).items()), 0 * a) / s[k]
                g = g + w[k] * (de[k][j] - 4 * G[k] * v)
                m = m + w[k] * (abs(de[k][j]) + 4 * Gm[k] * vm)
            out.append(g)
            mag.append(m)
    return np.stack(out, axis=1), np.stack(mag, axis=1)


def _jump(rng, quiet):
    side = (np.arange(5) < rng.integers(1, 5, (N, 1))) ^ (rng.random((N, 1)) < 0.5)
    return 1 + side * 10.0 ** rng.uniform(-2, 1, (N, 1)) + quiet * rng.random((N, 5))


FIELDS = {
    "jump": lambda r: _jump(r, 0.0),
    "jump_1e-9": lambda r: _jump(r, 1e-9),
    "jump_1e-3": lambda r: _jump(r, 1e-3),
    "noise": lambda r: 1 + r.random((N, 5)),
    "smooth": lambda r: 1.5 + np.sin(r.uniform(0, 6, (N, 1)) + 10.0 ** r.uniform(-4, -0.5, (N, 1)) * np.arange(5)),
    "scattered": lambda r: np.cumsum(10.0 ** r.uniform(-8, 1, (N, 5)) * r.choice([-1.0, 1.0], (N, 5)), axis=1),
}


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("field", sorted(FIELDS))
def test_derivatives_keep_their_own_scale(run, field, sign):
    q = sign * FIELDS[field](np.random.default_rng(9))
    o = run(q)
    want, mag = _exact(q)
    assert float(np.max(np.abs(o - want) / mag)) <= 32 * U
