"""GPU grid path with the gas + radiation EoS (Sect. 2.3, Eq. 6-7) against
the FP64 oracle, element by element, one step at a time.

The conserved state is read through Eq. 6 (e = rho R T/(gamma-1) + a T^4),
so with R = a = 1 the random test states have P_rad/P_gas between about 0.1
and 0.4.  Same bars as the ideal-gas parity tests: FP64 relative L1 per
component <= 1e-12 per step, FP32 <= 2e-5.
"""
import numpy as np
import pytest

import oracle as O
from paper_2503_04428_gb300 import workloads as wl

from parity import check
from test_parity_grid import step_compare

pytestmark = pytest.mark.gpu

RAD = (1.0, 1.0)  # R_gas, a_rad in code units


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("riemann", [O.HLL, O.HLLC])
def test_rad_1d(hydro_lib, precision, riemann):
    for ns, bc in ((0, (O.PERIODIC, O.PERIODIC)), (1, (O.TRANSMISSIVE, O.REFLECTIVE)), (3, (O.REFLECTIVE, O.TRANSMISSIVE))):
        case = wl.smooth_random(1, [600], ns, seed=21 + ns, bc=[bc], riemann=riemann)
        step_compare(hydro_lib, dict(case, eos_rad=RAD), precision, steps=2)


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("riemann", [O.HLL, O.HLLC])
def test_rad_2d(hydro_lib, precision, riemann):
    case = wl.smooth_random(2, [70, 37], 1, seed=5, riemann=riemann,
                            bc=[(O.PERIODIC, O.PERIODIC), (O.REFLECTIVE, O.TRANSMISSIVE)])
    step_compare(hydro_lib, dict(case, eos_rad=RAD), precision, steps=2)


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("ns", [0, 3])
def test_rad_3d(hydro_lib, precision, ns):
    case = wl.smooth_random(3, [37, 21, 35], ns, seed=9, riemann=O.HLLC,
                            bc=[(O.PERIODIC, O.PERIODIC), (O.TRANSMISSIVE, O.TRANSMISSIVE),
                                (O.REFLECTIVE, O.REFLECTIVE)])
    step_compare(hydro_lib, dict(case, eos_rad=RAD), precision, steps=2)


@pytest.mark.parametrize("precision", [64, 32])
def test_rad_spherical_3d(hydro_lib, precision):
    case = wl.sphere_state(nr=20, nth=12, nph=10, seed=13, riemann=O.HLLC, n_scalars=1,
                           ph_range=(0.0, 0.6))
    step_compare(hydro_lib, dict(case, eos_rad=RAD), precision, steps=2)


def test_rad_stationary_contact_stays_at_rest(hydro_lib):
    n = 300
    x = (np.arange(n) + 0.5) / n
    rho = np.where(x < 0.5, 1.0, 0.2)
    e = np.array([O.eos_rad_eint(5.0 / 3.0, 1.0, 1.0, r, 2.0)[1] for r in rho])
    U = np.stack([rho, np.zeros(n), e]).reshape(3, 1, 1, n)
    case = dict(name="contact", dim=1, n=[n, 1, 1], faces=[np.linspace(0, 1, n + 1)],
                bc=[(wl.PERIODIC, wl.PERIODIC)], coords=wl.CARTESIAN, gamma=5.0 / 3.0, n_scalars=0,
                riemann=wl.HLLC, limiter=wl.MINMOD, cfl=0.8, sources=None, U=U, eos_rad=(1.0, 1.0))
    g = hydro_lib.Grid.from_case(case, 64)
    g.run(50, 0.8)
    V = g.get_state()
    g.close()
    assert np.max(np.abs(V[1])) <= 1e-13
    assert np.max(np.abs(V - U)) <= 1e-12 * np.max(np.abs(U))


def test_rad_needs_hll_or_hllc(hydro_lib):
    case = wl.sod(64, riemann=wl.EXACT)
    g = hydro_lib.Grid.from_case(case, 64)
    with pytest.raises(hydro_lib.HydroError):
        g.set_eos_radiation(1.0, 1.0)
    g.close()


def _layers(axis, contrast, riemann, n=60):
    """Gas at rest in layers of three cells across `axis`, cold (T = 1) and hot (T = contrast) in turn: a radiation
    pressure that jumps by contrast^4 three planes on (n: the sweep takes several planes per CTA)."""
    i = np.arange(n) // 3 % 2
    T = np.where(i == 1, contrast, 1.0).reshape([n if d == axis else 1 for d in (2, 1, 0)]) * np.ones((n, n, n))
    U = np.zeros((5, n, n, n))
    U[0] = 1.0
    U[4] = T / (5.0 / 3.0 - 1.0) + T ** 4
    return dict(name="layers", dim=3, n=[n] * 3, faces=[np.linspace(0, 1, n + 1)] * 3, bc=[(wl.PERIODIC, wl.PERIODIC)] * 3,
                coords=wl.CARTESIAN, gamma=5.0 / 3.0, n_scalars=0, riemann=riemann, limiter=wl.MINMOD, cfl=0.4,
                sources=None, U=U, eos_rad=RAD)


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("riemann", [O.HLL, O.HLLC])
def test_rad_temperature_layers(hydro_lib, precision, riemann):
    """The new state's temperature is sought from the same cell's old one, whatever axis the temperature jumps along:
    after a step too short to move a layer, the signal speed is the oracle's, and the three orientations of the same
    layers take the same Newton iterations but for the cells that tiles and chunks stage twice (a fifth at most)."""
    its = []
    for axis in range(3):
        case = _layers(axis, 1000.0, riemann)
        if precision == 32:
            case["U"] = case["U"].astype(np.float32).astype(np.float64)
        s = O.solver_from_case(case)
        g = hydro_lib.Grid.from_case(case, precision)
        dt = 1e-9 * s.cfl_dt(0.4)
        s.step(dt)
        g.step(dt)
        assert g.cfl_dt(0.4) == pytest.approx(s.cfl_dt(0.4), rel=1e-12 if precision == 64 else 1e-5), axis
        its.append(g.stats()["newton_iters"])
        g.close()
    assert max(its) <= 1.2 * min(its), its


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("riemann", [O.HLL, O.HLLC])
def test_rad_cold_cells_heated_in_one_step(hydro_lib, precision, riemann):
    """Cold layers beside layers a thousand times hotter: one CFL step heats their edge cells by a factor of hundreds,
    and the temperature iteration, which starts at the cold value, has to arrive: the state and the next signal speed
    are the oracle's."""
    case = _layers(2, 1000.0, riemann, n=18)
    if precision == 32:
        case["U"] = case["U"].astype(np.float32).astype(np.float64)
    s = O.solver_from_case(case)
    g = hydro_lib.Grid.from_case(case, precision)
    dt = s.cfl_dt(0.4)
    s.step(dt)
    g.step(dt)
    check(s.get_state(), g.get_state(), 3, case["gamma"], precision)
    assert g.cfl_dt(0.4) == pytest.approx(s.cfl_dt(0.4), rel=1e-11 if precision == 64 else 1e-5)
    g.close()
