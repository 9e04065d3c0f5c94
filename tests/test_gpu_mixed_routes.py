"""Both routes of the mean stress in normal-mixed loading, each forced: summed from the stresses that
the two-pass residual has stored, and from the law again after the one-pass residual.  Bars as in
test_gpu_mixed.py, but for the FP32 iteration count, which its own tests hold."""

import numpy as np
import pytest

from abi_helpers import GpuProblem, rel_l2, sym6
from oracle.solver import Problem
from paper_2607_05929_gb300 import build
from paper_2607_05929_gb300 import fftm as F
from test_gpu_mixed import ALL_BUT_11, _two_phase

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("scheme", ["HEX1", "TETRA2"])
def test_both_routes_of_the_mean_stress_match_the_oracle(scheme, precision):
    build.build()
    F.load_library()
    tol = 1e-10 if precision == "fp64" else 1e-6
    wl = _two_phase(scheme, tol)
    pr = Problem(wl)
    _, rep = pr.solve_step(mixed=ALL_BUT_11)
    assert rep.converged
    ref = sym6(pr.last["P"])
    for passes in (1, 2):
        gp = GpuProblem(wl, precision)
        try:
            F.fftm_set_option(gp.p, F.FFTM_OPT_RESIDUAL_PASSES, passes)
            gp.set_load(wl.A, np.zeros(3), np.zeros((3, 6)), mixed=ALL_BUT_11)
            _, r, _, _ = F.fftm_solve_step(gp.p)
            assert r["converged"], passes
            if precision == "fp64":
                assert r["iterations"] == rep.iterations, passes
            A = F.fftm_get_load(gp.p)[0]
            assert np.abs(A - rep.A).max() < (1e-12 if precision == "fp64" else 1e-8), passes
            assert rel_l2(gp.get_voxel(F.FFTM_FIELD_STRESS), ref) < (1e-9 if precision == "fp64" else 1e-5), passes
        finally:
            gp.close()
