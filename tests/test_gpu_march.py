"""The stage kernel's walk along the radius at the sizes where its ring of rows, its groups of cells and
its teams change: the smallest instances, items of one cell (fewer cells than SMs), of two, of an odd count
and of the whole instance, items that start one or two cells from a wall; momentum sets of one warp (one
vector or two per thread), of a whole block (in FP32 also rows of eight per thread), and whose rows the bulk engine cannot copy (plain loads).
A cell's results do not depend on its item, so every tiling steps bit for bit alike; one of them is
compared with the oracle (the tolerances of the parity tests)."""
import numpy as np
import pytest

from oracle import solver as osolver
from paper_2403_15051_gb300 import build as fbuild
from paper_2403_15051_gb300 import fdlb
from paper_2403_15051_gb300 import workloads as wl

from .cases import compare_moments, oracle_problem, perturbed_state, small_case

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "fp32": 1e-5}


@pytest.fixture(scope="module", autouse=True)
def _built():
    fbuild.build()


SETS = [(wl.CYL, (4, 4, 4)), (wl.SPH, (4, 4, 4)), (wl.CYL, (4, 4, 8)), (wl.CYL, (3, 5, 3)), (wl.SPH, (5, 6, 4)),
        (wl.CYL, (8, 8, 8)), (wl.CYL, (9, 8, 8)), (wl.CYL, (1, 1, 1))]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("geom,Q", SETS)
@pytest.mark.parametrize("n_cells", [8, 11, 37])
def test_items_of_every_size_agree_and_match_oracle(n_cells, geom, Q, precision):
    d = small_case(geometry=geom, precision=precision, n_cells=n_cells, Q=Q, beta=1.0)
    P = oracle_problem(d)
    f0 = perturbed_state(P, 8, 0.05)
    # two instances: items of `cells` cells as asked (one instance alone is cut to fill the SMs)
    other = small_case(geometry=geom, precision=precision, n_cells=9, Q=Q)
    ref = None
    steps = 6 if min(Q) > 1 else 3  # (one node per axis: the oracle's own temperatures turn negative at the sixth)
    for cells in (None, 2, 3, 5, 64):
        with fdlb.Solver(d if cells is None else [d, other]) as S:
            S.set_autotune(0)
            if cells is not None:
                S.set_tiling(cells, 0, 0)
            S.set_f(f0, 0)
            S.step(steps)
            f = S.get_f(0)
            if ref is None:
                ref = f
                if min(Q) > 1:
                    errs = compare_moments(S.moments(0), osolver.moments(osolver.run(f0, P, steps), P), P)
                    assert max(errs.values()) <= TOL[precision], errs
            assert np.all(np.isfinite(f)) and np.array_equal(f, ref), cells


@pytest.mark.parametrize("Q", [(4, 4, 4), (4, 4, 8)])
def test_many_items_share_blocks(Q):
    # more items than SMs: several warps of a block walk items of their own, blocks take several items; a thread of
    # one vector, and of two (256 momenta over many cells)
    ds = [small_case(precision="fp32", n_cells=n, Q=Q, R=(1.0, 2.0 + 0.01 * q)) for q, n in enumerate([64, 33, 50] * 40)]
    out = []
    for cells in (2, 7, 64):
        with fdlb.Solver(ds) as S:
            S.set_autotune(0)
            S.set_tiling(cells, 0, 0)
            S.step(5)
            out.append([S.get_f(q) for q in (0, 1, 59, 119)])
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert np.all(np.isfinite(a)) and np.array_equal(a, b)
