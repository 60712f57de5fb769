"""States whose density jumps between neighbouring cells: the gradients of J1 take the logarithm of the ratio of
n^2 chi T, which must stay accurate (and finite) when that ratio is small.  The right-hand side of a perturbed
equilibrium with a step of 10, 100 and 1e4 in either direction against the oracle, with the tolerances of the
parity tests, in both forms of the closure.  A density that changes sign has no logarithm of a ratio: the right-hand
side there is not a number, so that a run from such a state reports it."""
import numpy as np
import pytest

from oracle import solver as osolver
from paper_2403_15051_gb300 import build as fbuild
from paper_2403_15051_gb300 import fdlb
from paper_2403_15051_gb300 import workloads as wl

from .cases import oracle_problem, perturbed_state, small_case

pytestmark = pytest.mark.gpu

RHS_TOL = {"fp64": 1e-10, "fp32": 2e-5}
N = 37


@pytest.fixture(scope="module", autouse=True)
def _built():
    fbuild.build()


def _rhs(d, f0, form):
    with fdlb.Solver(d) as S:
        assert S.closure_form(form) == form
        S.set_f(f0)
        return S.eval_rhs()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("geom", [wl.CYL, wl.SPH])
@pytest.mark.parametrize("chi_model", [fdlb.CHI_RET_FM, fdlb.CHI_SET_LOCAL])
@pytest.mark.parametrize("rising", [False, True])
@pytest.mark.parametrize("factor", [10.0, 100.0, 1e4])
def test_rhs_across_a_density_step_matches_oracle(factor, rising, chi_model, geom, precision):
    d = small_case(geometry=geom, precision=precision, n_cells=N, eta0=0.1, chi_model=chi_model)
    P = oracle_problem(d)
    step = np.where((np.arange(N) < N // 2) == rising, 1.0 / factor, 1.0)
    f0 = perturbed_state(P, 11, 0.05) * step[:, None, None, None]
    if precision == "fp32":
        f0 = f0.astype(np.float32).astype(np.float64)
    L_or = osolver.rhs(f0, P)
    for form in (0, 1):
        L = _rhs(d, f0, form)
        assert np.all(np.isfinite(L))
        assert np.max(np.abs(L - L_or)) <= RHS_TOL[precision] * np.max(np.abs(L_or)), form


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_a_negative_density_is_not_a_number(precision):
    d = small_case(precision=precision, n_cells=N)
    P = oracle_problem(d)
    f0 = perturbed_state(P, 11, 0.05)
    f0[N // 2] *= -1.0
    for form in (0, 1):
        assert np.any(np.isnan(_rhs(d, f0, form)[N // 2])), form
