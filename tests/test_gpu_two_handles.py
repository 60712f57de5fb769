"""Two handles in one process: a kernel's shared memory limit is the process's, so a handle on a smaller momentum
set, created or re-tiled between two steps of another, must not lower it under the other's launches."""
import numpy as np
import pytest

from paper_2403_15051_gb300 import build as fbuild
from paper_2403_15051_gb300 import fdlb

from .cases import small_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    fbuild.build()


def _wide(precision):
    # bands of more than 128 columns: the batch form of the closure launches its band kernel
    return [small_case(precision=precision, n_cells=300 + q, Q=(8, 8, 8)) for q in range(2)]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("form", [0, 1])
def test_a_smaller_handle_leaves_a_larger_one_stepping(form, precision):
    with fdlb.Solver(_wide(precision)) as A, fdlb.Solver(_wide(precision)) as B:
        for S in (A, B):
            S.set_autotune(0)
            assert S.closure_form(form) == form and S.info(0)["fm_band"] > 128
            S.step(1)
        with fdlb.Solver(small_case(precision=precision, n_cells=40, Q=(2, 2, 2))) as C:
            for change in (lambda: C.set_tiling(3, 0, 0), lambda: C.closure_form(1), lambda: C.set_closure_cells(3)):
                change()
                A.step(1)
                C.step(1)
        A.step(20)  # a graph
        B.step(23)
        for q in range(2):
            f = A.get_f(q)
            assert np.all(np.isfinite(f)) and np.array_equal(f, B.get_f(q))
