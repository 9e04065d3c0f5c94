"""The residual of crystal plasticity and logarithmic J2, whose stress kernel gives each voxel point
a thread of its own: tiles with remainders in x and y, fewer voxels than one tile and more than one,
both schemes, logarithmic J2 beside a Neo-Hookean phase, from a zero state past yield.

Tolerance, FP64: the laws' iterations end at 1e-12 of the largest stress and D is a sum of differences
of stresses of size |P| on a rough u^f (|D| ~ |P| / h); the slip's power n = 20 turns a unit of tau
into 20 of the slip increment: 1e-10.  FP32: the crystal law ends at two units of the largest stress
(2 * 6e-8), which n = 20 amplifies: 1e-5."""

import numpy as np
import pytest

import synthetic as syn
from abi_helpers import GpuProblem, rel_l2
from oracle.solver import Problem
from paper_2607_05929_gb300 import build
from paper_2607_05929_gb300 import fftm as F
from synthetic.workloads import CP_FCC, CP_FCC_PARAMS, LOG_J2, NEO_HOOKE, Material, Workload, axis_bc

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "fp32": 1e-5}
CP = [Material(CP_FCC, CP_FCC_PARAMS, tuple(q)) for q in syn.shoemake_quaternions(3, 9)]
LAWS = {
    "cp": (CP, 121.0, 49.25),
    "logj2": ([Material(LOG_J2, (1.2, 0.8, 2e-3)), Material(NEO_HOOKE, (0.1, 0.2))], 1.2, 0.8),
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    F.load_library()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("scheme", ["HEX1", "TETRA2"])
@pytest.mark.parametrize("laws", list(LAWS))
@pytest.mark.parametrize("n", [(2, 2, 2), (32, 8, 3), (36, 9, 4)])
def test_residual_matches_the_oracle(precision, scheme, laws, n):
    mats, lam0, mu0 = LAWS[laws]
    A = np.zeros((3, 3))
    A[0, 0] = 2e-3
    wl = Workload("points", n, syn.voronoi(n, len(mats), 6)[0], mats, axis_bc("D", "N", "P"), scheme=scheme,
                  lambda0=lam0, mu0=mu0, A=A)
    pr = Problem(wl)
    u = 5e-4 * np.random.default_rng(31).standard_normal(pr.grid.node_shape)
    for q in range(3):
        u[q][~pr.grid.dof_mask(q)] = 0.0
    if precision == "fp32":
        u = u.astype(np.float32).astype(np.float64)
    _, D_ref, _, _, SD, SP = pr.residual(u, pr.grad_ustar())
    gp = GpuProblem(wl, precision)
    try:
        gp.set_node(F.FFTM_FIELD_U, u)
        _, nm = F.fftm_apply(gp.p, F.FFTM_OP_RESIDUAL)
        D = gp.get_node(F.FFTM_FIELD_D)
    finally:
        gp.close()
    tol = TOL[precision]
    assert rel_l2(D, D_ref) < tol
    assert abs(nm[0] - SD) <= 10 * tol * SD
    assert abs(nm[1] - SP) <= tol * SP
