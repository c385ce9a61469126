"""Reciprocals, reciprocal square roots, sound speeds and quotients as the kernels form them (csrc/js_device.cuh),
with the GPU's own seeds, over every exponent that the integer forms take and mantissas beside powers of two.

Tolerance: a result of at least 56 correct bits rounded once, 2^-53 + 2^-56 relative (test_integer_weno.py checks
the same on the host, whose seeds are rounded differently)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cuda_runtime.h>
#include "js_device.cuh"
__global__ void eval(int op, int n, const double* a, const double* b, const double* c, double* o) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  if (op == 0) o[t] = js::recip(a[t]);
  else if (op == 1) o[t] = js::rsqrt_nr(a[t]);
  else if (op == 2) o[t] = js::sound(a[t], b[t], c[t]);
  else o[t] = js::quot_near(a[t], b[t], js::recip_top(js::mant64(b[t])));
}
extern "C" int wide_eval(int op, int n, const double* in, double* out) {
  double* d = nullptr;
  if (cudaMalloc(&d, sizeof(double) * 4 * n) != cudaSuccess) return 1;
  int rc = cudaMemcpy(d, in, sizeof(double) * 3 * n, cudaMemcpyHostToDevice) != cudaSuccess;
  if (!rc) {
    eval<<<(n + 255) / 256, 256>>>(op, n, d, d + n, d + 2 * n, d + 3 * n);
    rc = cudaMemcpy(out, d + 3 * n, sizeof(double) * n, cudaMemcpyDeviceToHost) != cudaSuccess;
  }
  cudaFree(d);
  return rc;
}
"""
LD = np.longdouble


@pytest.fixture(scope="module")
def wide(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("wide")
    (d / "t.cu").write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_04400_gb300", "csrc")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", inc, "-shared",
                    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", str(d / "t.cu"), "-o", str(d / "t.so")], check=True)
    f = ctypes.CDLL(str(d / "t.so")).wide_eval

    def run(op, *cols):
        x = np.ascontiguousarray(np.stack([np.broadcast_to(c, cols[0].shape) for c in cols + cols[:1] * (3 - len(cols))]))
        out = np.empty(x.shape[1])
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        assert f(op, x.shape[1], p(x), p(out)) == 0
        return out
    return run


def _mantissas(rng, n):
    m = 1.0 + rng.random(n)
    m[::5] = 1.0 + rng.integers(0, 40, m[::5].shape) * 2.0 ** -52
    m[1::5] = 2.0 - rng.integers(1, 40, m[1::5].shape) * 2.0 ** -52
    return m


def _check(got, want):
    assert float(np.max(np.abs(got - want) / np.abs(want))) <= 2.0 ** -53 + 2.0 ** -56


N = 400000


def test_reciprocals(wide):
    rng = np.random.default_rng(1)
    x = _mantissas(rng, N) * 2.0 ** rng.integers(-1022, 1022, N) * rng.choice([-1.0, 1.0], N)
    _check(wide(0, x), 1 / x.astype(LD))


def test_reciprocal_square_roots(wide):
    rng = np.random.default_rng(2)
    x = _mantissas(rng, N) * 2.0 ** rng.integers(-1022, 1023, N)
    _check(wide(1, x), 1 / np.sqrt(x.astype(LD)))


@pytest.mark.parametrize("reach", [4, 500, 1021])
def test_sound_speeds(wide, reach):
    rng = np.random.default_rng(3)
    g = 1.0 + 2.0 * rng.random(N)
    p, r = (_mantissas(rng, N) * 2.0 ** rng.integers(-reach, reach, N) for _ in range(2))
    _check(wide(2, g, p, r), np.sqrt(g.astype(LD) * p / r))


def test_quotients(wide):
    rng = np.random.default_rng(4)
    ea = rng.integers(-1000, 1000, N)
    eb = np.clip(ea + rng.integers(-1000, 1000, N), -1000, 1000)
    a = _mantissas(rng, N) * 2.0 ** ea * rng.choice([-1.0, 1.0], N)
    b = _mantissas(rng, N) * 2.0 ** eb * rng.choice([-1.0, 1.0], N)
    want = a.astype(LD) / b
    _check(wide(3, a, b), want)
    assert np.all(wide(3, np.zeros(8), b[:8]) == 0.0)
    with np.errstate(all="ignore"):  # outside the integer form's range: IEEE division
        a, b = np.array([1.0, 0.0, np.inf, 1e-310, 1e300, -3.0]), np.array([0.0, 0.0, 2.0, 3.0, 1e-300, 1e-310])
        assert np.array_equal(wide(3, a, b), a / b, equal_nan=True)
