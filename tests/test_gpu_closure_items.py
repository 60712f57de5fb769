"""The closure's items at the sizes where their shapes change: the smallest instances, item counts
that divide the cells unevenly, bands of up to 64, up to 128 and more columns (summed by the records
kernel eight or four rows at a time, or by the band kernel), enough cells for the widest items, and
the chain form with band rows that do not fit in a block's share of shared memory.  The records do not
depend on the grouping, so every grouping steps bit for bit like the chain form with items of two
cells (itself compared with the oracle elsewhere)."""
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


def _states_after(ds, states, steps, cells=None):
    with fdlb.Solver(ds) as S:
        S.set_autotune(0)
        if cells is None:
            assert S.closure_form(1) == 1
        else:
            S.set_closure_cells(cells)
        widest = max(S.info(q)["fm_band"] for q in range(len(ds)))
        for q, f in enumerate(states):
            S.set_f(f, q)
        S.step(steps)
        return widest, [S.get_f(q) for q in range(len(ds))]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("geom,Q", [(wl.CYL, (4, 4, 4)), (wl.SPH, (3, 5, 5))])
@pytest.mark.parametrize("cells,lo,hi", [((8, 12, 13, 29), 0, 64), ((120, 57), 65, 128), ((240, 8), 129, 1000)])
def test_batch_form_equals_the_chain_at_item_and_band_edges(cells, lo, hi, geom, Q, precision):
    ds = [small_case(geometry=geom, precision=precision, n_cells=n, Q=Q, R=(1.0, 2.0 + 0.1 * q), Kn=0.08)
          for q, n in enumerate(cells)]
    states = [perturbed_state(oracle_problem(d), 3 + q, 0.05) for q, d in enumerate(ds)]
    widest, ref = _states_after(ds, states, 5, cells=2)
    assert lo <= widest <= hi
    for other in (None, 7, 28):
        _, got = _states_after(ds, states, 5, cells=other)
        for a, b in zip(ref, got):
            assert np.all(np.isfinite(a)) and np.array_equal(a, b), other


def test_wide_items_and_throughput_chain_equal_the_small_items():
    # 36000 cells: 28-cell items in the batch form; in the chain form more items than blocks, the band rows
    # beyond a block's share of shared memory read from global memory
    ds = [small_case(precision="fp32", n_cells=1000, Q=(2, 2, 2), R=(1.0, 2.0 + 0.05 * q), Kn=0.06) for q in range(36)]
    out = []
    for cells in (2, 8, 16, None):
        with fdlb.Solver(ds) as S:
            S.set_autotune(0)
            if cells is None:
                assert S.closure_form(1) == 1
            else:
                S.set_closure_cells(cells)
            S.step(4)
            out.append([S.get_f(q) for q in (0, 17, 35)])
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert np.all(np.isfinite(a)) and np.array_equal(a, b)
