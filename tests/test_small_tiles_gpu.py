"""The small 1D and 2D tiles of the general sweep (csrc/sweep.cuh, small_tile) at their edges.

One step against the oracle, at the per-step bars of tests/parity.py: grids
of fewer tiles than the GPU has SMs, at and around multiples of the tiles (28
cells in 1D, 8 x 8 in 2D), with every solver, precision and scalar count, and
a grid on either side of the rule that picks the tile.
"""
import numpy as np
import pytest

import oracle as O
from paper_2503_04428_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

from parity import check

P, T, R = O.PERIODIC, O.TRANSMISSIVE, O.REFLECTIVE


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("n", [[2], [27], [28], [29], [57], [1000], [200000], [2, 2], [7, 9], [8, 8], [9, 17], [64, 33],
                               [400, 300]])
def test_sizes(hydro_lib, n, precision):
    for k, riemann in enumerate((O.HLL, O.HLLC, O.EXACT)):
        if np.prod(n) > 10000 and k != len(n):
            continue
        bc = [[(P, P)] * 2, [(T, R), (R, T)], [(R, R), (T, T)]][(k + n[0]) % 3][:len(n)]
        case = wl.smooth_random(len(n), n, (k + n[0]) % 4, seed=80 + k, bc=bc, riemann=riemann,
                                limiter=[O.MINMOD, O.VANLEER, O.VANALBADA][k])
        case["U"] = case["U"].astype(np.float32).astype(np.float64)
        ref = O.solver_from_case(case)
        dt = ref.cfl_dt(0.4)
        ref.step(dt)
        g = hydro_lib.Grid.from_case(case, precision)
        g.set_step_totals(True)
        g.step(dt)
        check(ref.get_state(), g.get_state(), len(n), case["gamma"], precision)
        tot = g.totals()
        assert np.allclose(g.step_totals(), tot, rtol=0, atol=1e-6 * np.abs(tot).max())
        g.close()
