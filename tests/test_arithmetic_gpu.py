"""The FP64 reciprocal, quotient and square root of the step (csrc/physics.cuh) against correctly rounded ones.

They are steps of their own from the PTX approximations, so they are checked as the operators they stand for: over the
exponents that their comments state, at random and extreme mantissas, equal to the correctly rounded results (numpy's
division and square root) or next to them, with an error of at most half a unit in the last place and 2^-20 of one.
"""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "physics.cuh"
using namespace hydro;
__global__ void run(int what, const double* a, const double* b, double* r, long n) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i < n) r[i] = what == 0 ? rcp<double>(a[i]) : what == 1 ? qdiv<double>(a[i], b[i]) : dsqrt<double>(a[i]);
}
extern "C" int apply(int what, const double* a, const double* b, double* r, long n) {
  double* d = nullptr;
  const size_t s = n * sizeof(double);
  if (cudaMalloc(&d, 3 * s) != cudaSuccess) return 1;
  cudaMemcpy(d, a, s, cudaMemcpyHostToDevice);
  cudaMemcpy(d + n, b, s, cudaMemcpyHostToDevice);
  run<<<(unsigned)((n + 255) / 256), 256>>>(what, d, d + n, d + 2 * n, n);
  const int e = cudaMemcpy(r, d + 2 * n, s, cudaMemcpyDeviceToHost) != cudaSuccess;
  cudaFree(d);
  return e;
}
"""


@pytest.fixture(scope="module")
def apply(hydro_lib, tmp_path_factory):
    from paper_2503_04428_gb300 import build
    d = tmp_path_factory.mktemp("arithmetic")
    src, so = str(d / "probe.cu"), str(d / "probe.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.NVCC] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, "-shared", "-cudart", "shared", src, "-o", so],
                   check=True, cwd=os.path.dirname(src))
    lib = ctypes.CDLL(so)

    def call(what, a, b=None):
        a = np.ascontiguousarray(a, dtype=np.float64)
        b = np.ones_like(a) if b is None else np.ascontiguousarray(b, dtype=np.float64)
        r = np.empty_like(a)
        p = [x.ctypes.data_as(ctypes.c_void_p) for x in (a, b, r)]
        assert lib.apply(what, *p, ctypes.c_long(a.size)) == 0
        return r
    return call


def _numbers(rng, n, lo, hi):
    """n numbers with exponents in [lo, hi]: random mantissas, and ones next to 1 and 2."""
    m = 1.0 + rng.random(n)
    edge = np.array([1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 1.5, 4 / 3, 1.0 + 2.0 ** -20 - 2.0 ** -52, 1.0 + 2.0 ** -32])
    m[:n // 8] = edge[rng.integers(0, len(edge), n // 8)]
    return np.ldexp(m, rng.integers(lo, hi + 1, n))


def _compare(got, want, error):
    """error(result, k): the exact error of a result for argument k, over that argument's exact result."""
    off = np.nonzero(got != want)[0]
    assert off.size <= got.size // 20
    for k in off[:: max(1, off.size // 2000)]:
        g, w = Fraction(float(got[k])), float(want[k])
        assert abs(error(g, k)) * abs(Fraction(w)) <= Fraction(float(np.spacing(abs(w)))) * (Fraction(1, 2) + Fraction(1, 2 ** 20)), k


@pytest.mark.parametrize("exponents", [(-1, 1), (-100, 100), (-1022, 1020)])
def test_reciprocal(apply, exponents):
    rng = np.random.default_rng(1)
    x = _numbers(rng, 1 << 20, *exponents) * rng.choice([-1.0, 1.0], 1 << 20)
    _compare(apply(0, x), 1.0 / x, lambda r, k: r * Fraction(float(x[k])) - 1)


@pytest.mark.parametrize("exponents", [(-1, 1), (-100, 100), (-500, 500)])
def test_quotient(apply, exponents):
    rng = np.random.default_rng(2)
    a = _numbers(rng, 1 << 20, *exponents) * rng.choice([-1.0, 1.0], 1 << 20)
    b = _numbers(rng, 1 << 20, *exponents) * rng.choice([-1.0, 1.0], 1 << 20)
    for a, b in ((a, b), (_numbers(rng, 1 << 18, -1000, -900), _numbers(rng, 1 << 18, -1020, -900)),
                 (_numbers(rng, 1 << 18, 900, 1020), _numbers(rng, 1 << 18, 900, 1020))):
        _compare(apply(1, a, b), a / b, lambda r, k: r * Fraction(float(b[k])) / Fraction(float(a[k])) - 1)
    assert np.all(apply(1, np.zeros(3), np.array([1.0, -2.0, 1e300])) == 0.0)


@pytest.mark.parametrize("exponents", [(-2, 2), (-100, 100), (-1000, 1023)])
def test_square_root(apply, exponents):
    x = _numbers(np.random.default_rng(3), 1 << 20, *exponents)
    # (r^2/x - 1 = 2 e + e^2 for a relative error e)
    _compare(apply(2, x), np.sqrt(x), lambda r, k: (r * r / Fraction(float(x[k])) - 1) / 2)
    assert np.all(apply(2, np.array([0.0, -0.0])) == 0.0)


def test_exact_solver_takes_a_side_without_pressure(hydro_lib):
    """P = 0 on one side: its sound speed is 0, and the star state is that of the shock into it,
    (p - p_R) sqrt(2/((g + 1) rho_R p)) = u_R + ... : p* solves f_L(p) + f_R(p) + du = 0."""
    g = 1.4
    WL, WR = np.array([[1.0, 0.0, 1.0], [2.0, 1.0, 3.0]]), np.array([[1.0, 0.0, 0.0], [0.5, -1.0, 0.0]])
    ps, us, _ = hydro_lib.hydro_exact_solve(WL, WR, g)
    for k in range(2):
        p, (rL, uL, pL), (rR, uR, _) = ps[k], WL[k], WR[k]
        c = np.sqrt(g * pL / rL)
        fL = ((p - pL) * np.sqrt(2 / ((g + 1) * rL) / (p + (g - 1) / (g + 1) * pL)) if p > pL
              else 2 * c / (g - 1) * ((p / pL) ** ((g - 1) / (2 * g)) - 1))
        fR = np.sqrt(2 * p / ((g + 1) * rR))
        assert p > 0 and abs(fL + fR + uR - uL) <= 1e-12 * (abs(fL) + fR)
        assert abs(us[k] - (uR + fR)) <= 1e-12 * (abs(uR) + fR)
