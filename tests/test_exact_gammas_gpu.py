"""The exact solver's roots (csrc/physics.cuh, pow_z) for every gamma it treats as one, and for gammas it does not.

Star states of random faces against the oracle's: FP64 to 1e-11 relative (a
root correct to a few ulp, eps = 1.1e-16, moves p* by at most the condition
of the face, below 1e4 at the 5 % vacuum margin kept here), FP32 to the 5e-6
that the FP32 star pressure keeps, of faces given at FP32's gamma.
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma", [4 / 3, 1.4, 1.5, 5 / 3, 2.0, 1.25, 1.6, 3.0])
@pytest.mark.parametrize("precision", [64, 32])
def test_star_states(hydro_lib, gamma, precision):
    rng = np.random.default_rng(int(1000 * gamma))
    n = 400
    g = gamma if precision == 64 else float(np.float32(gamma))
    span = 8.0 if precision == 64 else 5.0
    W = [np.stack([10.0 ** rng.uniform(-3, 3, n), rng.uniform(-2, 2, n), 10.0 ** rng.uniform(-span / 2, span / 2, n)], 1)
         for _ in range(2)]
    if precision == 32:
        W = [w.astype(np.float32).astype(np.float64) for w in W]
    WL, WR = W
    c = [np.sqrt(g * w[:, 2] / w[:, 0]) for w in W]
    vac = 2 / (g - 1) * (c[0] + c[1])
    keep = WR[:, 1] - WL[:, 1] < (0.95 if precision == 64 else 0.8) * vac
    WL, WR = WL[keep], WR[keep]
    ps, us, _ = hydro_lib.hydro_exact_solve(WL, WR, gamma, precision=precision)
    tol = 1e-11 if precision == 64 else 5e-6
    cmax = np.maximum(*c)[keep]
    for k in range(len(ps)):
        p, u = O.exact_star(g, WL[k], WR[k])[:2]
        assert abs(ps[k] - p) <= tol * p, (k, ps[k], p)
        assert abs(us[k] - u) <= tol * max(abs(u), cmax[k]), (k, us[k], u)


@pytest.mark.parametrize("gamma", [1.3333333333, 1.3333333334, 1.6666666667, 1.6666666666, 1.40000000003, 1.5 + 1e-11,
                                   2.0 - 1e-10, 1.4 + 2e-14])
def test_gammas_next_to_a_root(hydro_lib, gamma):
    """FP64 star states at gammas whose 1/z is nearly, but not, an integer:
    the powers have to be those of the gamma given, to the same 1e-11."""
    states = [((1.0, 0.0, 1.0), (0.125, 0.0, 0.1)), ((1.0, -2.0, 0.4), (1.0, 2.0, 0.4)),
              ((1.0, -1.0, 1e3), (2.0, 1.0, 1e-2)), ((3.0, 0.5, 2.0), (1.0, 0.9, 1.9))]
    W = [np.array([s[k] for s in states]) for k in range(2)]
    c = [np.sqrt(gamma * w[:, 2] / w[:, 0]) for w in W]
    keep = W[1][:, 1] - W[0][:, 1] < 0.95 * 2 / (gamma - 1) * (c[0] + c[1])  # (the second is a vacuum at gamma = 2)
    W = [w[keep] for w in W]
    ps, us, _ = hydro_lib.hydro_exact_solve(W[0], W[1], gamma)
    for k in range(len(ps)):
        p, u = O.exact_star(gamma, W[0][k], W[1][k])[:2]
        assert abs(ps[k] - p) <= 1e-11 * p, (k, ps[k], p)
        assert abs(us[k] - u) <= 1e-11 * max(abs(u), np.sqrt(gamma * W[0][k, 2] / W[0][k, 0])), (k, us[k], u)
