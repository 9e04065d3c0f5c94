"""The residual's form is chosen among what was compared: a problem that is held to one pass (and
compares its tiles alone) leaves no choice behind for one that may take two, nor does a problem of
another law of the same shape."""

import numpy as np
import pytest

from abi_helpers import GpuProblem
from paper_2607_05929_gb300 import build
from paper_2607_05929_gb300 import fftm as F
from synthetic.workloads import CUBIC_ELASTIC, ISO_ELASTIC, Material, Workload, axis_bc

pytestmark = pytest.mark.gpu

N = (18, 8, 6)  # a shape that no other test solves on


def _solve(material, passes):
    A = np.zeros((3, 3))
    A[0, 0] = 1e-3
    wl = Workload("tuning", N, np.zeros(N, dtype=np.int32), [material], axis_bc("D", "N", "P"), scheme="HEX1",
                  lambda0=121.0, mu0=49.25, A=A)
    gp = GpuProblem(wl, "fp64", tol=1e-6)
    try:
        F.fftm_set_option(gp.p, F.FFTM_OPT_RESIDUAL_PASSES, passes)
        assert F.fftm_solve_step(gp.p)[1]["converged"]
    finally:
        gp.close()
    return [t for t in F.fftm_tuning_table().splitlines() if "HEX1 %dx%dx%d BBP" % N in t]


def test_each_choice_names_what_it_compared():
    build.build()
    F.load_library()
    iso, cubic = Material(ISO_ELASTIC, (60.0, 40.0)), Material(CUBIC_ELASTIC, (168.0, 121.0, 75.0))
    one = _solve(iso, 1)
    assert len(one) == 1 and "two passes" not in one[0]
    both = [t for t in _solve(iso, 0) if t not in one]
    assert len(both) == 1 and "two passes" in both[0], both
    assert len(_solve(iso, 0)) == 2  # the choice is kept
    assert len(_solve(cubic, 0)) == 3
