"""Batches stepped as two chains of launches (the halves of the instances): every instance as in a handle of
its own, bit for bit, in graphs and direct launches, beside the single chain of the timing mode, with bands wide
enough for the band kernel, and with an instance that retires under a captured graph."""
import numpy as np
import pytest

from paper_2403_15051_gb300 import build as fbuild
from paper_2403_15051_gb300 import fdlb
from paper_2403_15051_gb300 import workloads as wl

from .cases import oracle_problem, perturbed_state, small_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    fbuild.build()


def _alone(d, f, advance):
    with fdlb.Solver(d) as S:
        S.set_autotune(0)
        S.set_f(f)
        advance(S)
        return S.get_f()


@pytest.mark.parametrize("geom,Q,cells,batch_form", [
    (wl.CYL, (8, 8, 8), (29, 8, 64, 13, 40), False), (wl.CYL, (8, 8, 8), (240, 9), True), (wl.SPH, (12, 12, 12), (12, 8, 9), False)])
def test_lanes_equal_single_instances(geom, Q, cells, batch_form):
    # (on a dozen cells between spheres the step from the CFL number is unstable: the oracle's too)
    ds = [small_case(geometry=geom, precision="fp32", n_cells=n, Q=Q, R=(1.0, 2.0 + 0.1 * q), Kn=0.08,
                     dt=1e-3 if geom == wl.SPH else None) for q, n in enumerate(cells)]
    states = [perturbed_state(oracle_problem(d), 3 + q, 0.05) for q, d in enumerate(ds)]

    def advance(S):
        S.step(1)
        S.step(23)  # a graph of 20 and three direct

    with fdlb.Solver(ds) as S:
        S.set_autotune(0)
        if batch_form:
            assert max(S.info(q)["fm_band"] for q in range(len(ds))) > 128 and S.closure_form(1) == 1
        for timing in (False, True):
            for q, f in enumerate(states):
                S.set_f(f, q)
            S.set_kernel_timing(timing)
            advance(S)
            for q, (d, f) in enumerate(zip(ds, states)):
                got, ref = S.get_f(q), _alone(d, f, advance)
                assert np.all(np.isfinite(got)) and np.array_equal(got, ref), (timing, q)


def test_lanes_with_a_retired_instance():
    # the second instance is at rest between equal walls: it retires at the first check, with 25 steps to go
    ds = [small_case(precision="fp32", n_cells=n, Q=(8, 8, 8), R=(1.0, 2.0), Kn=0.08, **kw)
          for n, kw in ((24, {}), (30, dict(T_wall=(1.0, 1.0), u_wall=(0.0, 0.0), eta0=0.01)), (16, {}))]
    states = [perturbed_state(oracle_problem(d), 3 + q, 0.05) for q, d in enumerate(ds)]
    run = lambda S: S.run_to_steady(tol=1e-4, max_steps=75, check_every=25)  # noqa: E731
    with fdlb.Solver(ds) as S:
        S.set_autotune(0)
        S.set_f(states[0], 0)
        S.set_f(states[2], 2)
        _, steps, _ = run(S)
        assert steps[1] < 75 and steps[0] == steps[2] == 75
        for q in (0, 2):
            assert np.array_equal(S.get_f(q), _alone(ds[q], states[q], run)), q
