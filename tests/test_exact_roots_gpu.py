"""The FP64 powers of the exact solver as roots (csrc/physics.cuh, pow_z and behind_fan), to a fraction of an ulp.

x^z with z = 1/n, and rho q^(1/gamma) behind a rarefaction of pressure ratio q, for the gammas whose n is 4 to 8, over the
ratios that the solver meets (Newton's floor is 1e-14): the estimate is good to 1e-6 there, so one third-order step leaves
n^2/12 1e-18 < 0.05 ulp, the correction's own rounding less, and the final rounding 0.5: 0.6 allowed.  The density is one
rounding of a quotient whose divisor carries twice the root's 0.1: 0.8.  Reference: extended precision.
"""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "physics.cuh"
using namespace hydro;
__global__ void run(const double* x, double* t, double* rho, long n, Gas<double> gas) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  t[i] = pow_z(x[i], gas);
  double same;
  rho[i] = behind_fan(x[i + n], x[i], gas, same);
  if (same != t[i]) rho[i] = -1.0;
}
extern "C" int roots(int root, double gamma, const double* x, double* out, long n) {
  double* d = nullptr;
  if (cudaMalloc(&d, 4 * n * sizeof(double)) != cudaSuccess) return 1;
  cudaMemcpy(d, x, 2 * n * sizeof(double), cudaMemcpyHostToDevice);
  Gas<double> g{};
  g.root = root;
  g.z = 1.0 / root;
  g.ig = 1.0 / gamma;
  run<<<(unsigned)((n + 127) / 128), 128>>>(d, d + 2 * n, d + 3 * n, n, g);
  const int e = cudaMemcpy(out, d + 2 * n, 2 * n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess;
  cudaFree(d);
  return e;
}
"""


@pytest.fixture(scope="module")
def roots(hydro_lib, tmp_path_factory):
    from paper_2503_04428_gb300 import build
    d = tmp_path_factory.mktemp("roots")
    (d / "probe.cu").write_text(SOURCE)
    subprocess.run([build.NVCC] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, "-shared", "-cudart", "shared",
                                                              str(d / "probe.cu"), "-o", str(d / "probe.so")], check=True)
    return ctypes.CDLL(str(d / "probe.so"))


@pytest.mark.parametrize("n", [4, 5, 6, 7, 8])
def test_roots(roots, n):
    gamma = n / (n - 2.0)  # 1/z = 2 gamma/(gamma - 1) = n
    rng, m = np.random.default_rng(n), 1 << 17
    q = np.concatenate([10.0 ** rng.uniform(-14, 0, m), 1.0 - 10.0 ** rng.uniform(-15, -1, m), 10.0 ** rng.uniform(0, 8, m)])
    r = 10.0 ** rng.uniform(-3, 3, q.size)
    x, out = np.concatenate([q, r]), np.empty(2 * q.size)
    vp = ctypes.c_void_p
    assert roots.roots(n, ctypes.c_double(gamma), x.ctypes.data_as(vp), out.ctypes.data_as(vp), ctypes.c_long(q.size)) == 0
    t, rho = out[:q.size], out[q.size:]
    X = np.longdouble
    root = X(q) ** (X(1) / n)
    for got, want, ulps in ((t, root, 0.6), (rho, X(r) * (X(q) / (root * root)), 0.8)):
        e = np.abs(X(got) - want) / np.spacing(np.abs(want.astype(np.float64)))
        assert np.all(e <= ulps), (n, float(e.max()), q[np.argmax(e)])
