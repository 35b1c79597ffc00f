"""The HLL flux (csrc/physics.cuh; csrc/pair.cuh for the FP32 march) of slow, nearly uniform flow.

The mass and scalar fluxes a rho_L u_L + b rho_R u_R + c (rho_L - rho_R) of its formula (c = S_L S_R/(S_R - S_L) the
dissipation) are small there against rho c, and their error has to be small against their own terms: a dozen roundings of
|a rho_L u_L| + |b rho_R u_R| + |c (rho_L - rho_R)| (the wave speeds, the quotient, the factors and the sums; for the
scalar, the products rho f as well, whose rounding the difference keeps: c rho f).  Reference: the same formula in
extended precision on the same states and sound speeds.
"""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pair.cuh"
using namespace hydro;
// states (rho, u, p, f) x 2 per face; out: the flux and the two sound speeds
__global__ void run64(const double* w, double* f, long n, Gas<double> gas) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double *L = w + 8 * i, *R = L + 4;
  double e, cL, cR;
  face_e_c<double>(gas, L[0], L[2], 0.0, e, cL);
  face_e_c<double>(gas, R[0], R[2], 0.0, e, cR);
  hll_flux<double, 1, 1, 0>(L, R, L[2] * gas.igm1, R[2] * gas.igm1, cL, cR, f + 6 * i);
  f[6 * i + 4] = cL;
  f[6 * i + 5] = cR;
}
__global__ void run32(const double* w, double* f, long n, Gas<float> g) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Gas2 gas(g);
  f2 L[4], R[4], F[4];
  for (int v = 0; v < 4; ++v) {
    L[v] = both((float)w[8 * i + v]);
    R[v] = both((float)w[8 * i + 4 + v]);
  }
  hll2<1, 1, 0>(L, R, F, gas);
  for (int v = 0; v < 4; ++v) f[6 * i + v] = (double)(i % 2 ? hi(F[v]) : lo(F[v]));
  f[6 * i + 4] = (double)lo(sound2(L[0], L[2], gas));
  f[6 * i + 5] = (double)lo(sound2(R[0], R[2], gas));
}
extern "C" int fluxes(int precision, const double* w, double* f, long n) {
  double* d = nullptr;
  if (cudaMalloc(&d, 14 * n * sizeof(double)) != cudaSuccess) return 1;
  cudaMemcpy(d, w, 8 * n * sizeof(double), cudaMemcpyHostToDevice);
  const unsigned blocks = (unsigned)((n + 127) / 128);
  Gas<double> g64{};
  g64.g = 1.4;
  g64.gm1 = 1.4 - 1.0;
  g64.igm1 = 1.0 / (1.4 - 1.0);
  Gas<float> g32{};
  g32.g = (float)g64.g;
  g32.gm1 = (float)g64.gm1;
  g32.igm1 = (float)g64.igm1;
  if (precision == 64) run64<<<blocks, 128>>>(d, d + 8 * n, n, g64);
  else run32<<<blocks, 128>>>(d, d + 8 * n, n, g32);
  const int e = cudaMemcpy(f, d + 8 * n, 6 * n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess;
  cudaFree(d);
  return e;
}
"""


@pytest.fixture(scope="module")
def fluxes(hydro_lib, tmp_path_factory):
    from paper_2503_04428_gb300 import build
    d = tmp_path_factory.mktemp("hll")
    (d / "probe.cu").write_text(SOURCE)
    subprocess.run([build.NVCC] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, "-shared", "-cudart", "shared",
                                                              str(d / "probe.cu"), "-o", str(d / "probe.so")], check=True)
    lib = ctypes.CDLL(str(d / "probe.so"))

    def call(precision, w):
        f = np.empty((len(w), 6))
        assert lib.fluxes(precision, w.ctypes.data_as(ctypes.c_void_p), f.ctypes.data_as(ctypes.c_void_p),
                          ctypes.c_long(len(w))) == 0
        return f
    return call


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("du,drho", [(1e-1, 1e-1), (1e-3, 1e-4), (1e-6, 0.0), (1e-6, 1e-5), (3.0, 0.5)])
def test_mass_and_scalar_flux(fluxes, precision, du, drho):
    rng, n = np.random.default_rng(5), 20000
    dt = np.float64 if precision == 64 else np.float32
    w = np.empty((n, 2, 4))
    w[:, :, 0] = rng.uniform(0.5, 2.0, (n, 1)) * (1 + drho * rng.uniform(-1, 1, (n, 2)))
    w[:, :, 1] = du * rng.uniform(-1, 1, (n, 2))
    w[:, :, 2] = rng.uniform(0.5, 2.0, (n, 2))
    w[:, :, 3] = rng.uniform(0.0, 1.0, (n, 1)) * (1 + drho * rng.uniform(-1, 1, (n, 2)))
    w = np.ascontiguousarray(w.astype(dt).astype(np.float64))
    f = fluxes(precision, w.reshape(n, 8))
    X = np.longdouble
    (rL, uL, _, sL), (rR, uR, _, sR) = [[X(w[:, k, v]) for v in range(4)] for k in range(2)]
    cL, cR = X(f[:, 4]), X(f[:, 5])
    SL, SR = np.minimum(np.minimum(uL - cL, uR - cR), 0), np.maximum(np.maximum(uL + cL, uR + cR), 0)
    a, b, c = SR / (SR - SL), -SL / (SR - SL), SL * SR / (SR - SL)
    eps = 2.0 ** -53 if precision == 64 else 2.0 ** -24
    for v, (qL, qR), products in ((0, (rL, rR), 0.0), (3, (rL * sL, rR * sR), 1.0)):
        want = a * uL * qL + b * uR * qR + c * (qR - qL)
        size = np.abs(a * uL * qL) + np.abs(b * uR * qR) + np.abs(c * (qR - qL))
        bound = 12 * eps * (size + products * np.abs(c) * (qL + qR) / 12) * (1 if precision == 64 else 2)
        assert np.all(np.abs(X(f[:, v]) - want) <= bound), (v, float((np.abs(X(f[:, v]) - want) / bound).max()))
