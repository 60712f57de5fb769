"""Applying a handle's own configuration again (the tuner's candidates, a cached choice, the setters of other
options) keeps the stage kernel: the same momenta per thread and vectors, so the same order of the moment sums
and the same bits.  Momentum sets on either side of the rules that choose the kernel: rows of eight p_2 momenta
with one warp per cell, the reduced pair, a block that holds one vector of four or would hold two, FP64."""
import numpy as np
import pytest

from oracle import solver as osolver
from paper_2403_15051_gb300 import build as fbuild
from paper_2403_15051_gb300 import fdlb
from paper_2403_15051_gb300 import workloads as wl

from .cases import compare_moments, oracle_problem, perturbed_state, small_case

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


# (set, precision, cells, threads asked for, the most that may come of it: what the vectors of two FP64 or four FP32
# momenta, four or two to a thread, took)
BLOCKS = [(wl.SPH, (12, 12, 12), "fp32", 20, 256, 224), (wl.SPH, (12, 12, 12), "fp32", 20, 288, 288),
          (wl.CYL, (8, 8, 4), "fp64", 24, 64, 64), (wl.CYL, (8, 8, 4), "fp64", 24, 128, 128), (wl.CYL, (4, 4, 4), "fp64", 24, 32, 32),
          (wl.CYL, (4, 4, 8), "fp64", 24, 64, 64), (wl.SPH, (4, 4, 4), "fp64", 24, 32, 32), (wl.CYL, (4, 8, 4), "fp32", 24, 32, 32),
          (wl.CYL, (9, 8, 8), "fp32", 24, 160, 160), (wl.CYL, (8, 8, 8), "fp64", 24, 256, 256)]


@pytest.mark.parametrize("geometry,Q,precision,cells,threads,most", BLOCKS)
def test_the_block_size_asked_for_is_kept(geometry, Q, precision, cells, threads, most):
    d = small_case(geometry=geometry, precision=precision, n_cells=cells, Q=Q)
    P = oracle_problem(d)
    f0 = perturbed_state(P, 8, 0.05)
    with fdlb.Solver(d) as S:
        S.set_tiling(0, 0, threads)
        assert S.tiling()["threads"] <= most
        S.set_tiling(0, 0, 0)
        S.set_tensor_contraction(False)
        assert S.tiling()["threads"] <= most
        S.set_f(f0)
        L, L_or = S.eval_rhs(), osolver.rhs(f0, P)
        assert np.max(np.abs(L - L_or)) <= (1e-10 if precision == "fp64" else 2e-5) * np.max(np.abs(L_or))
        S.step(2)
        errs = compare_moments(S.moments(), osolver.moments(osolver.run(f0, P, 2), P), P)
        assert max(errs.values()) <= (1e-10 if precision == "fp64" else 1e-5), errs


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_the_cells_per_tile_asked_for_are_kept_on_a_lone_instance(precision):
    # 64 cells in one tile are walked by one block, cell after cell: many times the stage's time over the default,
    # a cell to an item, and the same bits
    d = small_case(precision=precision, n_cells=64, Q=(4, 4, 4))
    out = {}
    for cells in (0, 64):
        with fdlb.Solver(d) as S:
            S.set_tiling(cells, 0, 0)
            S.step(5)
            out[cells] = S.get_f()
            S.set_kernel_timing(True)
            S.step(20)
            out[cells, "ms"] = S.kernel_times()[0]
    assert np.array_equal(out[0], out[64])
    assert out[64, "ms"] > 4.0 * out[0, "ms"]
