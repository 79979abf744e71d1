"""The pair sum's reciprocal square root (an estimate and one Halley step)
over every r^2 that a neighbour list can hold, whatever the unit of length.

FP64, against exact rational arithmetic: the last addition rounds (2^-53
relative), and the residual e = 1 - r^2 y^2 carries the rounding of r^2 y
(2^-53), halved: below 2^-52 in all.  r = r^2 (1/r) rounds once more: below
2^-52 + 2^-53, and CUDA's own sqrt and division stand beside it.  FP32 likewise
with 2^-24: below 2^-23 and 2^-23 + 2^-24.

The FP64 mobility in a unit of length in which a bead's radius is 1e-21 (and
1e-23) must be the one at radius 1 scaled: 1e-12 relative, as for two
evaluations of the same sums with other rounding."""

import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "fsd_internal.cuh"
template <typename T>
__global__ void k(int n, const T *r2, T *out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const T y = fsd::inv_sqrt<T>(r2[i]);
  out[3 * i] = y;
  out[3 * i + 1] = r2[i] * y;
  out[3 * i + 2] = sqrt(r2[i]);
}
template <typename T>
static int go(int n, const T *r2, T *out) {
  T *a = nullptr, *b = nullptr;
  if (cudaMalloc(&a, n * sizeof(T)) != cudaSuccess || cudaMalloc(&b, 3 * n * sizeof(T)) != cudaSuccess) return 1;
  cudaMemcpy(a, r2, n * sizeof(T), cudaMemcpyHostToDevice);
  k<T><<<(n + 127) / 128, 128>>>(n, a, b);
  const cudaError_t e = cudaMemcpy(out, b, 3 * n * sizeof(T), cudaMemcpyDeviceToHost);
  cudaFree(a);
  cudaFree(b);
  return e != cudaSuccess;
}
extern "C" int run64(int n, const double *r2, double *out) { return go(n, r2, out); }
extern "C" int run32(int n, const float *r2, float *out) { return go(n, r2, out); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2607_25161_gb300 import build

    d = tmp_path_factory.mktemp("inv_sqrt")
    (d / "t.cu").write_text(SOURCE)
    so = str(d / "t.so")
    r = subprocess.run([build.nvcc(), "-O3", "-std=c++17", build.ARCH, "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
                        "-shared", "-I", build.SRC, "-I", os.path.join(ROOT, "include"), "-o", so, str(d / "t.cu")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


@pytest.mark.parametrize("dtype,name,lo,hi,u", [(np.float64, "run64", -298, 298, 2.0 ** -53),
                                                (np.float32, "run32", -36, 37, 2.0 ** -24)])
def test_inverse_distance_over_its_range(lib, dtype, name, lo, hi, u):
    rng = np.random.default_rng(4)
    r2 = np.concatenate([10.0 ** rng.uniform(lo, hi, 6000), 10.0 ** rng.uniform(-2, 4, 6000),
                         4.0 * (1.0 + np.arange(-200, 200) * 4 * u)]).astype(dtype)
    out = np.empty((len(r2), 3), dtype)
    assert getattr(lib, name)(len(r2), r2.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p)) == 0
    worst = [0.0, 0.0, 0.0]
    for x, (y, r, root) in zip(r2, out):
        f, yy, rr = Fraction(float(x)), Fraction(float(y)), Fraction(float(r))
        # y sqrt(x) - 1 = (x y^2 - 1) / 2 to first order; r / sqrt(x) - 1 likewise
        worst[0] = max(worst[0], abs(float(f * yy * yy - 1)) / 2)
        worst[1] = max(worst[1], abs(float(rr * rr / f - 1)) / 2)
        worst[2] = max(worst[2], abs(float(Fraction(float(root)) ** 2 / f - 1)) / 2)
    assert worst[2] <= u * 1.0001  # CUDA's sqrt rounds correctly
    assert worst[0] <= 2 * u and worst[1] <= 3 * u, worst


@pytest.mark.parametrize("unit", [1e-3, 1e-21, 1e-23])
def test_fp64_mobility_in_any_unit_of_length(unit):
    import __graft_entry__ as g
    import paper_2607_25161_gb300 as pkg

    g.build()
    rng = np.random.default_rng(6)
    pos = rng.uniform(0.0, 16.0, size=(24, 3))
    F = np.zeros((24, 11))
    F[:, :3] = rng.normal(size=(24, 3))
    u = {}
    for a in (1.0, unit):
        s = pkg.Suspension(pos * a, np.arange(24), 16.0 * a, a=a, xi=0.9 / a, rc=6.5 * a, grid=32, P=8,
                           restart=2, inner_restart=2)
        u[a] = s.apply_mobility(F)[:, :3] * a
        s.close()
    assert np.linalg.norm(u[unit] - u[1.0]) <= 1e-12 * np.linalg.norm(u[1.0])
