"""The residual of small-strain laws on the strain alone, where its branches meet: isotropic and
cubic phases in one problem (the law read per voxel) and each by itself (one law for the kernel),
a quadratic mean field, unequal spacings, one pass (both tiles) and two, FP32 and FP64.

Tolerance: D is a sum of differences of stresses of size |P|, and on a rough u^f |D| ~ |P| / h, so
that a handful of roundings per stress entry (the sums, six products, the differences) stay below
16 units: 16 * 6e-8 = 1e-6 in FP32; 1e-12 in FP64 leaves 4 digits more than that count needs."""

import numpy as np
import pytest

import synthetic as syn
from abi_helpers import GpuProblem, rel_l2
from oracle.solver import Problem
from paper_2607_05929_gb300 import build
from paper_2607_05929_gb300 import fftm as F
from synthetic.workloads import CUBIC_ELASTIC, ISO_ELASTIC, Material, Workload, axis_bc

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-6}
CUBIC = [Material(CUBIC_ELASTIC, (168.0, 121.0, 75.0), tuple(v)) for v in syn.shoemake_quaternions(2, 8)]
ISO = [Material(ISO_ELASTIC, (60.0, 40.0)), Material(ISO_ELASTIC, (110.0, 75.0))]
LAWS = {"iso": ISO, "cubic": CUBIC, "both": [ISO[0], CUBIC[0], CUBIC[1], ISO[1]]}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    F.load_library()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("scheme", ["HEX1", "TETRA2"])
@pytest.mark.parametrize("laws", list(LAWS))
@pytest.mark.parametrize("n", [(36, 12, 8), (32, 9, 18)])
def test_residual_matches_the_oracle(precision, scheme, laws, n):
    mats = LAWS[laws]
    A = np.array([[1e-3, -2e-4, 0.0], [3e-4, 5e-4, 0.0], [-4e-4, 1e-4, 0.0]])
    Q = np.zeros((3, 6))
    Q[0, 0], Q[1, 1], Q[2, 5] = 2e-5, -3e-5, 1e-5  # second-order in x and y only: z is periodic
    wl = Workload("strain", n, syn.voronoi(n, len(mats), 6)[0], mats, axis_bc("D", "N", "P"), scheme=scheme,
                  lambda0=90.0, mu0=55.0, h=(1.0, 0.75, 1.3), A=A, Q=Q)
    pr = Problem(wl)
    u = 1e-3 * np.random.default_rng(21).standard_normal(pr.grid.node_shape)
    for q in range(3):
        u[q][~pr.grid.dof_mask(q)] = 0.0
    if precision == "fp32":
        u = u.astype(np.float32).astype(np.float64)
    _, D_ref, _, _, SD, SP = pr.residual(u, pr.grad_ustar())
    tol = TOL[precision]
    for passes, tile in ((1, 8), (1, 16), (2, 0)):
        gp = GpuProblem(wl, precision)
        try:
            F.fftm_set_option(gp.p, F.FFTM_OPT_RESIDUAL_PASSES, passes)
            F.fftm_set_option(gp.p, F.FFTM_OPT_RESIDUAL_TILE, tile)
            gp.set_node(F.FFTM_FIELD_U, u)
            _, nm = F.fftm_apply(gp.p, F.FFTM_OP_RESIDUAL)
            D = gp.get_node(F.FFTM_FIELD_D)
        finally:
            gp.close()
        assert rel_l2(D, D_ref) < tol, (passes, tile)
        assert abs(nm[0] - SD) <= 10 * tol * SD, (passes, tile)
        assert abs(nm[1] - SP) <= tol * SP, (passes, tile)
