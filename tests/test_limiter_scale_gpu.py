"""The FP32 smooth limiters (csrc/physics.cuh) on states of very small density.

Every conserved variable times 2^-80 (densities of 1e-24) leaves speeds and
limiter ratios as they are and scales the step's result by the same power of
two, so one step of the scaled state, scaled back, meets the oracle's step of
the unscaled one at the per-step bars of tests/parity.py: a limiter that
multiplied two slopes would find 0 there.
"""
import numpy as np
import pytest

import oracle as O
from paper_2503_04428_gb300 import workloads as wl
from parity import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limiter", [O.VANLEER, O.VANALBADA])
@pytest.mark.parametrize("n", [(37,), (29, 7), (13, 9, 5)])
def test_small_densities(hydro_lib, n, limiter):
    case = wl.smooth_random(len(n), list(n), 1, seed=7, bc=[(O.PERIODIC, O.PERIODIC)] * len(n), riemann=O.HLLC,
                            limiter=limiter)
    case["U"] = case["U"].astype(np.float32).astype(np.float64)
    ref = O.solver_from_case(case)
    dt = ref.cfl_dt(0.4)
    ref.step(dt)
    g = hydro_lib.Grid.from_case(dict(case, U=case["U"] * 2.0**-80), 32)
    g.step(dt)
    check(ref.get_state(), g.get_state() * 2.0**80, case["dim"], case["gamma"], 32)
    g.close()


@pytest.mark.parametrize("riemann", [O.HLL, O.HLLC, O.EXACT])
@pytest.mark.parametrize("n", [(37,), (29, 17), (13, 9, 5)])
def test_subnormal_densities_end_in_an_error(hydro_lib, n, riemann):
    """Densities of 2^-127 (subnormal in FP32, whose reciprocals take them for 0): the step reports a failure and leaves
    the state, and does not go on from wrong velocities."""
    case = wl.smooth_random(len(n), list(n), 1, seed=7, bc=[(O.PERIODIC, O.PERIODIC)] * len(n), riemann=riemann)
    g = hydro_lib.Grid.from_case(case, 32)
    dt = g.cfl_dt(0.4)
    U = (case["U"] * 2.0**-127).astype(np.float32)
    g.set_state(U)
    with pytest.raises(hydro_lib.HydroError) as e:
        g.step(dt)
    assert e.value.status in (hydro_lib.HYDRO_ERR_NEGATIVE_STATE, hydro_lib.HYDRO_ERR_NONFINITE, hydro_lib.HYDRO_ERR_NEWTON,
                              hydro_lib.HYDRO_ERR_VACUUM)
    assert np.array_equal(g.get_state(), U)
    g.close()
