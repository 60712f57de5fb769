"""Applying a handle's own configuration again (the tuner's candidates, a cached choice, the setters of other
options) keeps the stage kernel: the same momenta per thread and vectors, so the same order of the moment sums
and the same bits.  Momentum sets on either side of the rules that choose the kernel: rows of eight p_2 momenta
with one warp per cell, the reduced pair, a block that holds one vector of four or would hold two, FP64."""
import numpy as np
import pytest

from paper_2403_15051_gb300 import build as fbuild
from paper_2403_15051_gb300 import fdlb
from paper_2403_15051_gb300 import workloads as wl

from .cases import small_case

pytestmark = pytest.mark.gpu

KERNEL = ("threads", "slice_k", "stage_vector_width", "stage_vectors_per_thread")


@pytest.fixture(scope="module", autouse=True)
def _built():
    fbuild.build()


def _batch(geometry, Q, precision, cells):
    return [small_case(geometry=geometry, precision=precision, n_cells=n, Q=Q, R=(1.0, 2.0 + 0.2 * q))
            for q, n in enumerate(cells)]


def _kernel(S):
    t = S.tiling()
    return tuple(t[k] for k in KERNEL)


# (more than 8 cells per SM, where one warp takes two vectors of four, and fewer)
MANY, FEW = (700, 650, 301), (70, 65, 31)
SETS = [(wl.CYL, (4, 8, 4), "fp32", MANY), (wl.CYL, (4, 8, 4), "fp32", FEW), (wl.CYL_Z, (8, 8, 0), "fp32", MANY),
        (wl.CYL, (5, 8, 4), "fp32", MANY), (wl.CYL, (9, 8, 8), "fp32", FEW), (wl.CYL, (4, 4, 8), "fp32", MANY),
        (wl.CYL, (4, 8, 4), "fp64", MANY), (wl.SPH, (4, 8, 4), "fp32", MANY), (wl.CYL, (8, 8, 8), "fp32", MANY)]


@pytest.mark.parametrize("geometry,Q,precision,cells", SETS)
def test_tuning_keeps_the_kernel_and_every_bit(geometry, Q, precision, cells):
    ds = _batch(geometry, Q, precision, cells)
    with fdlb.Solver(ds) as A, fdlb.Solver(ds) as B, fdlb.Solver(ds) as C:
        A.set_autotune(0)
        made = _kernel(A)
        B.autotune()
        for S in (A, B, C):  # untuned, tuned, and with the cached choice
            S.step(5)
            assert _kernel(S) == made
        for q in range(len(ds)):
            f = A.get_f(q)
            assert np.all(np.isfinite(f))
            assert np.array_equal(f, B.get_f(q)) and np.array_equal(f, C.get_f(q)), q


@pytest.mark.parametrize("geometry,Q,precision,cells", SETS)
def test_setters_of_other_options_keep_the_kernel(geometry, Q, precision, cells):
    with fdlb.Solver(_batch(geometry, Q, precision, cells)) as S:
        made = _kernel(S)
        for change in (lambda: S.set_tensor_contraction(False), lambda: S.set_persistent_step(False),
                       lambda: S.stage_min_blocks(1), lambda: S.set_tiling(5, 0, 0), lambda: S.set_tiling(0, 0, 0)):
            change()
            assert _kernel(S) == made
