"""fdlb_set_tensor_contraction at 2Q_R = 32 .. 48 radial nodes, where the stage contracts K^h itself by default: the
contraction kernel can be selected in both precisions (a third launch per stage; on the tensor cores in FP32, on
the CUDA cores in FP64, which is not reported as in use) and taken back, and either way matches the oracle with
the tolerances of the parity tests."""
import numpy as np
import pytest

from oracle import solver as osolver
from paper_2403_15051_gb300 import build as fbuild
from paper_2403_15051_gb300 import fdlb
from paper_2403_15051_gb300 import workloads as wl

from .cases import oracle_problem, perturbed_state, small_case

pytestmark = pytest.mark.gpu

RHS_TOL = {"fp64": 1e-10, "fp32": 2e-5}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("geom,Q", [(wl.CYL, (16, 4, 4)), (wl.CYL, (24, 8, 4)), (wl.SPH, (20, 4, 4))])
def test_the_contraction_kernel_can_be_selected(geom, Q, precision):
    fbuild.build()
    d = small_case(geometry=geom, precision=precision, n_cells=21, Q=Q, beta=0.8, Kn=0.05, eta0=0.15)
    P = oracle_problem(d)
    f0 = perturbed_state(P, 17, 0.05)
    L_or = osolver.rhs(f0, P)
    with fdlb.Solver(d) as S:
        for enable, launches in ((None, 6), (True, 9), (False, 6)):
            if enable is not None:
                assert bool(S.set_tensor_contraction(enable)) == (enable and precision == "fp32")
            S.set_f(f0)
            assert np.max(np.abs(S.eval_rhs() - L_or)) <= RHS_TOL[precision] * np.max(np.abs(L_or)), enable
            S.step(1)
            assert S.launch_count() == launches, enable
