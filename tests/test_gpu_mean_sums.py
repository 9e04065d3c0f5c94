"""The mean stress and gradient of a step's report are sums of FP64's precision whatever the fields'.

u_3 rises in four steps along z, at one (x, y) node alone, so that four columns of voxels hold the
normal stress (lambda = 0, 2 mu = 1) and gradient 33 of a quarter of each step, and nothing else does.
The steps lie 38 planes apart: where 608 blocks walk 32 x 8 tiles of 64 x 64 voxels, one thread meets
all four of a column.  The levels 0, t, 1 + 2^-23, -1, 3 with t = 2^-28 + 2^-51 give steps that FP32
rounds to t, 1 + 2^-23, -2, 4: their sum, 3 + 2^-23 + 2^-28 + 2^-51, takes 53 bits, every partial sum
and every sum of the columns is exact in FP64, and so is the mean over 2^19 voxels."""

import numpy as np
import pytest

from abi_helpers import GpuProblem
from paper_2607_05929_gb300 import build
from paper_2607_05929_gb300 import fftm as F
from synthetic.workloads import ISO_ELASTIC, Material, Workload, axis_bc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp32_tf32", "fp64"])
def test_means_keep_every_bit_of_an_fp64_sum(precision):
    build.build()
    F.load_library()
    n = (64, 64, 128)
    wl = Workload("steps", n, np.zeros(n, dtype=np.int32), [Material(ISO_ELASTIC, (0.0, 0.5))],
                  axis_bc("N", "N", "N"), scheme="HEX1", lambda0=0.0, mu0=0.5)
    gp = GpuProblem(wl, precision, tol=1e30)
    try:
        u = np.zeros((3,) + gp.N)
        for z, level in ((2, 2.0 ** -28 + 2.0 ** -51), (40, 1 + 2.0 ** -23), (78, -1.0), (116, 3.0)):
            u[2, 20, 11, z:] = level
        gp.set_node(F.FFTM_FIELD_U, u)
        _, rep, _, _ = F.fftm_solve_step(gp.p)  # at rest at once: the report of the field given
    finally:
        gp.close()
    assert rep["iterations"] == 0
    d = np.diff(u[2, 20, 11])
    steps = d if precision == "fp64" else d.astype(np.float32)
    total = float(np.sum(steps.astype(np.longdouble)))
    assert precision == "fp64" or total == 3 + 2.0 ** -23 + 2.0 ** -28 + 2.0 ** -51
    assert rep["mean_P"][2] * 2.0 ** 19 == total
    assert rep["mean_G"][8] * 2.0 ** 19 == total
