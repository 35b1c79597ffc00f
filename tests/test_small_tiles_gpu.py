"""The small 1D and 2D tiles of the general sweep (csrc/sweep.cuh, small_tile) at their edges.

One step against the oracle, at the per-step bars of tests/parity.py: grids
of fewer tiles than the GPU has SMs, at and around multiples of the tiles (28
cells in 1D, 8 x 8 in 2D), with every solver, precision and scalar count, and
a grid on either side of the rule that picks the tile.
"""
import time

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


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("n", [[2], [29], [300], [4000], [3, 5], [40, 33], [120, 100]])
def test_run_equals_single_steps(hydro_lib, n, precision):
    """hydro_run (many steps in one launch on these grids) against the same
    steps one by one with hydro_cfl_dt, to the rounding of the steps: 12 steps
    of at most ~100 roundings, eps = 1.1e-16 / 6e-8, allowing a factor of 30
    for the flow's growth; and the time clipped to t_end, a run past it doing
    nothing more."""
    for k, riemann in enumerate((O.HLL, O.HLLC, O.EXACT)):
        case = wl.smooth_random(len(n), n, k + 1, seed=90 + k, bc=[(T, R), (P, P)][:len(n)], riemann=riemann)
        a, b = [hydro_lib.Grid.from_case(case, precision) for _ in range(2)]
        for _ in range(12):
            b.step(b.cfl_dt(0.4))
        t = a.run(12, 0.4)
        sb = b.stats()
        assert a.stats()["steps"] == sb["steps"] == 12
        tol = 3e-13 if precision == 64 else 2e-4
        assert abs(t - sb["t"]) <= tol * sb["t"]
        A, B = a.get_state().astype(np.float64), b.get_state().astype(np.float64)
        assert np.abs(A - B).max() <= tol * np.abs(B).max()
        t_end = t + 1.5 * a.stats()["last_dt"]
        assert a.run(100, 0.4, t_end) == pytest.approx(t_end, rel=1e-14)
        done = a.stats()["steps"]
        assert 13 <= done <= 15
        a.run(7, 0.4, t_end)
        assert a.stats()["steps"] == done
        a.close()
        b.close()


@pytest.mark.parametrize("n", [[200], [40, 24]])
def test_failed_run_keeps_the_last_good_state(hydro_lib, n):
    """A run at a hopeless CFL number fails after some steps: status, step
    count and state are those of the last good step, and the handle goes on."""
    case = wl.smooth_random(len(n), n, 0, seed=5, amp=0.5, riemann=O.HLLC)
    a, b = [hydro_lib.Grid.from_case(case, 64) for _ in range(2)]
    good = 0
    with pytest.raises(hydro_lib.HydroError) as e1:
        for _ in range(60):
            b.step(b.cfl_dt(6.0))
            good += 1
    with pytest.raises(hydro_lib.HydroError) as e2:
        a.run(60, 6.0)
    assert e1.value.status == e2.value.status
    assert a.stats()["steps"] == good and a.stats()["t"] == pytest.approx(b.stats()["t"], rel=1e-9)
    A, B = a.get_state(), b.get_state()
    assert np.abs(A - B).max() <= 1e-6 * np.abs(B).max()
    a.run(3, 0.2)
    assert a.stats()["steps"] == good + 3
    a.close()
    b.close()


@pytest.mark.parametrize("n", [[4000], [100, 90]])
def test_failure_in_the_first_step_ends_the_run_at_once(hydro_lib, n):
    """A first step that fails in one corner of the grid ends a many-step run without any CTA waiting out its bound (4
    million polls, seconds), however late the others start: a hundred runs, each of milliseconds (a tenth of a second
    allowed), each leaving the state as it was."""
    case = wl.smooth_random(len(n), n, 0, seed=5, amp=0.01, riemann=O.HLLC, bc=[(T, T)] * len(n))
    case["U"][1, ..., :2] = -30.0 * case["U"][0, ..., :2]  # two columns torn off
    case["U"][-1, ..., :2] += 0.5 * 900.0 * case["U"][0, ..., :2]
    g = hydro_lib.Grid.from_case(case, 64)
    U = g.get_state()
    for _ in range(100):
        t = time.perf_counter()
        with pytest.raises(hydro_lib.HydroError) as e:
            g.run(50, 5.0)
        assert time.perf_counter() - t < 0.1
        assert e.value.status in (hydro_lib.HYDRO_ERR_NEGATIVE_STATE, hydro_lib.HYDRO_ERR_NONFINITE)
        assert g.stats()["steps"] == 0 and np.array_equal(g.get_state(), U)
    g.close()


@pytest.mark.parametrize("n", [[20], [500], [40, 24]])
def test_an_expired_wait_loses_the_state(hydro_lib, n):
    """A many-step run whose waits expire (bound 0: no word is ever seen) reports HYDRO_ERR_TIMEOUT, and since its CTAs
    may have ended at different steps, every call that needs the state refuses until one is set; then the handle works."""
    H = hydro_lib
    case = wl.smooth_random(len(n), n, 0, seed=5, riemann=O.HLLC)
    g = H.Grid.from_case(case, 64)
    g.set_step_wait(0)
    with pytest.raises(H.HydroError) as e:
        g.run(10, 0.4)
    assert e.value.status == H.HYDRO_ERR_TIMEOUT and "wait" in str(e.value)
    for call in (lambda: g.run(1, 0.4), lambda: g.step(1e-6), g.get_state, lambda: g.cfl_dt(0.4), g.totals,
                 lambda: g.get_boundary(0, 0)):
        with pytest.raises(H.HydroError) as e:
            call()
        assert e.value.status == H.HYDRO_ERR_TIMEOUT
    g.set_step_wait(1 << 22)
    g.set_state(case["U"])
    steps = g.stats()["steps"]
    assert np.array_equal(g.get_state(), case["U"].reshape(g.shape))
    g.run(10, 0.4)
    assert g.stats()["steps"] == steps + 10
    with pytest.raises(H.HydroError):
        g.set_step_wait(-1)
    g.close()


def _sourced(kind, n):
    if kind == "point":
        case = wl.sphere_state(*n, n_scalars=1, dim=len(n), riemann=O.HLLC)
        case["sources"] = dict(gravity=O.GRAV_POINT, G=3.0, Mc=2.0)
    elif kind == "const":
        case = wl.smooth_random(len(n), n, 1, seed=33, riemann=O.HLL, bc=[(T, R), (P, P)][:len(n)])
        case["sources"] = dict(gravity=O.GRAV_UNIFORM, g0=(0.3, -0.2, 0.0), heating=O.HEAT_CONST, heat_params=(50.0,))
    else:  # Ni-56 in CGS units on a grid of 1e14 cm: a run spans days, over which the heating decays
        case = wl.smooth_random(len(n), n, 2, seed=34, riemann=O.HLLC, bc=[(T, R), (P, P)][:len(n)])
        case["faces"] = [1e14 * np.asarray(f) for f in case["faces"]]
        x = np.linspace(0, 1, n[0])[None, None, :] * np.ones((1, n[1] if len(n) > 1 else 1, 1))
        vel = [1e7 * np.sin(4 * x)] + [np.zeros_like(x)] * (len(n) - 1)
        case["U"] = wl.conserved(case["gamma"], 1e-9 * (1 + 0.3 * np.sin(6 * x)), vel, 1e5 * (1 + 0.2 * np.cos(5 * x)),
                                 [np.full_like(x, 0.5), 0.1 + 0.05 * np.sin(3 * x)])
        case["sources"] = dict(heating=O.HEAT_NI56, heat_params=(1,))
    return case


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("n", [[300], [40, 33]])
@pytest.mark.parametrize("kind", ["point", "const", "ni56"])
def test_run_with_sources_equals_single_steps(hydro_lib, kind, n, precision):
    """Gravity and heating in a many-step run, which keeps the time (and so the Ni-56 heating's decay) itself, against
    single steps, at the bars of test_run_equals_single_steps; and without the sources the run ends elsewhere."""
    case = _sourced(kind, n)
    a, b, c = [hydro_lib.Grid.from_case(dict(case, sources=s), precision) for s in (case["sources"], case["sources"], None)]
    for g in (a, b, c):
        g.set_time(86400.0 * 5 if kind == "ni56" else 0.0)
    t = a.run(12, 0.4)
    c.run(12, 0.4)
    for _ in range(12):
        b.step(b.cfl_dt(0.4))
    sa, sb = a.stats(), b.stats()
    tol = 3e-13 if precision == 64 else 2e-4
    assert sa["steps"] == sb["steps"] == 12 and abs(t - sb["t"]) <= tol * sb["t"]
    A, B, C = [g.get_state().astype(np.float64) for g in (a, b, c)]
    for v in range(len(A)):
        assert np.abs(A[v] - B[v]).max() <= tol * max(np.abs(B[v]).max(), 1e-3 * np.abs(B[0]).max() if kind != "ni56" else 0)
    e = 1 + len(n)
    assert np.abs(A[e] - C[e]).max() > 100 * tol * np.abs(A[e]).max()  # the sources act
    if kind == "ni56":
        assert t - 86400.0 * 5 > 0.5 * 86400  # (of a decay time of 8.8 days)
    for g in (a, b, c):
        g.close()
