"""The FP32 marching steps (csrc/march3.cuh, march2.cuh) at the edges of their tiles, halves and chunks.

One step of each grid against the oracle, at the per-step bars of
tests/parity.py: sizes at and around the owned columns of a warp (30) and the
owned rows of a CTA (14, 10 and 8 for 0, 1 and 2-3 scalars) in 3D, the owned
columns of a warp (28) and the longest run of rows (2 x 64) in 2D, the
smallest axes, odd counts (the high half of a pair then misses its last plane
or row), every boundary kind and both coordinate systems; and repeated runs
give the same bits.
"""
import numpy as np
import pytest

import oracle as O
from paper_2503_04428_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

from parity import check

P, T, R = O.PERIODIC, O.TRANSMISSIVE, O.REFLECTIVE
SIZES = [(2, 2, 2), (29, 13, 3), (30, 14, 4), (31, 15, 5), (61, 29, 7), (3, 10, 9), (60, 11, 2), (32, 8, 33),
         (91, 9, 6), (5, 43, 11)]
BCS = [[(P, P)] * 3, [(T, R), (R, T), (P, P)], [(R, R), (P, P), (T, R)], [(T, T), (T, T), (R, T)]]


@pytest.mark.parametrize("k", range(len(SIZES)))
@pytest.mark.parametrize("ns", [0, 1, 2, 3])
def test_cartesian_sizes(hydro_lib, k, ns):
    case = wl.smooth_random(3, list(SIZES[k]), ns, seed=40 + k, bc=BCS[(k + ns) % 4],
                            riemann=[O.HLL, O.HLLC][(k + ns) % 2], limiter=[O.MINMOD, O.VANLEER, O.VANALBADA][k % 3])
    _one_step(hydro_lib, case)


@pytest.mark.parametrize("n", [(2, 2, 2), (31, 11, 5), (30, 8, 9)])
@pytest.mark.parametrize("riemann", [O.HLL, O.HLLC])
def test_spherical_sizes(hydro_lib, n, riemann):
    case = wl.sphere_state(*n, n_scalars=3, dim=3, riemann=riemann)
    case["sources"] = dict(gravity=O.GRAV_POINT_MONOPOLE, G=0.01, Mc=2.0)
    _one_step(hydro_lib, case)


SIZES2 = [(2, 2), (27, 3), (28, 4), (29, 5), (57, 64), (3, 131), (84, 129), (30, 257)]


@pytest.mark.parametrize("k", range(len(SIZES2)))
@pytest.mark.parametrize("ns", [0, 1, 2, 3])
def test_2d_sizes(hydro_lib, k, ns):
    case = wl.smooth_random(2, list(SIZES2[k]), ns, seed=60 + k, bc=BCS[(k + ns) % 4][:2],
                            riemann=[O.HLL, O.HLLC][(k + ns) % 2], limiter=[O.MINMOD, O.VANLEER, O.VANALBADA][k % 3])
    case["sources"] = dict(gravity=O.GRAV_UNIFORM, g0=(0.1, -0.2, 0.0))
    _one_step(hydro_lib, case)


@pytest.mark.parametrize("n", [(2, 2), (29, 7), (56, 130)])
@pytest.mark.parametrize("riemann", [O.HLL, O.HLLC])
def test_2d_spherical_sizes(hydro_lib, n, riemann):
    case = wl.sphere_state(*n, n_scalars=1, dim=2, riemann=riemann)
    case["sources"] = dict(gravity=O.GRAV_POINT, G=0.01, Mc=2.0)
    _one_step(hydro_lib, case)


def _one_step(hydro_lib, case):
    case["U"] = case["U"].astype(np.float32).astype(np.float64)
    ref = O.solver_from_case(case)
    dt = ref.cfl_dt(0.4)
    ref.step(dt)
    out = []
    for _ in range(2):
        g = hydro_lib.Grid.from_case(case, 32)
        g.set_step_totals(True)
        g.step(dt)
        check(ref.get_state(), g.get_state(), case["dim"], case["gamma"], 32)
        g.run(4, 0.4)
        out.append((g.get_state(), g.step_totals()))
        g.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


# sizes that the march takes (march3_pays), at and around its tiles' edges, with odd and remaining planes
MARCHED = [(150, 70, 33), (119, 39, 81), (209, 83, 45), (211, 85, 46), (600, 40, 21), (299, 23, 35), (60, 8, 300),
           (30, 300, 40), (149, 55, 150), (600, 420, 7), (1200, 2, 40), (899, 3, 31), (2, 3, 4100)]


@pytest.mark.parametrize("k", range(len(MARCHED)))
@pytest.mark.parametrize("ns", [0, 1, 2, 3])
def test_cartesian_sizes_that_march(hydro_lib, k, ns):
    case = wl.smooth_random(3, list(MARCHED[k]), ns, seed=70 + k, bc=BCS[(k + ns) % 4],
                            riemann=[O.HLL, O.HLLC][(k + ns) % 2], limiter=[O.MINMOD, O.VANLEER, O.VANALBADA][k % 3])
    _marches(hydro_lib, case)
    _one_step(hydro_lib, case)


@pytest.mark.parametrize("n", [(150, 70, 33), (299, 23, 35), (601, 41, 21)])
@pytest.mark.parametrize("riemann", [O.HLL, O.HLLC])
@pytest.mark.parametrize("ns", [0, 1, 3])
def test_spherical_sizes_that_march(hydro_lib, n, riemann, ns):
    case = wl.sphere_state(*n, n_scalars=ns, dim=3, riemann=riemann)
    case["sources"] = dict(gravity=O.GRAV_POINT_MONOPOLE, G=0.01, Mc=2.0)
    _marches(hydro_lib, case)
    _one_step(hydro_lib, case)


def _marches(hydro_lib, case):
    g = hydro_lib.Grid.from_case(case, 32)
    g.run(1, 0.4)
    assert g.stats()["tile_x"] == 30  # (the general sweep's tiles are 16 wide)
    g.close()
