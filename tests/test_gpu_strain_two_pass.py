"""The two-pass residual of small-strain laws on the strain alone (k_stress, k_div) against the oracle,
on a caller's field.  FFTM_OP_RESIDUAL with two passes forms p as well and takes the kernels with test
outputs; fftm_residual_noalloc runs the solver's own once a step has settled the form.  Workload and
tolerances as in test_gpu_strain_path.py."""

import numpy as np
import pytest

import synthetic as syn
from abi_helpers import GpuProblem, node_from_abi, node_to_abi, rel_l2
from oracle.solver import Problem
from paper_2607_05929_gb300 import build
from paper_2607_05929_gb300 import fftm as F
from synthetic.workloads import Workload, axis_bc
from test_gpu_strain_path import LAWS, TOL

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("scheme", ["HEX1", "TETRA2"])
@pytest.mark.parametrize("laws", list(LAWS))
def test_two_pass_residual_matches_the_oracle(precision, scheme, laws):
    build.build()
    F.load_library()
    mats, n = LAWS[laws], (36, 12, 8)
    A = np.array([[1e-3, -2e-4, 0.0], [3e-4, 5e-4, 0.0], [-4e-4, 1e-4, 0.0]])
    Q = np.zeros((3, 6))
    Q[0, 0], Q[1, 1], Q[2, 5] = 2e-5, -3e-5, 1e-5
    wl = Workload("strain", n, syn.voronoi(n, len(mats), 6)[0], mats, axis_bc("D", "N", "P"), scheme=scheme,
                  lambda0=90.0, mu0=55.0, h=(1.0, 0.75, 1.3), A=A, Q=Q)
    pr = Problem(wl)
    gp = GpuProblem(wl, precision, tol=1e30)
    try:
        u = 1e-3 * np.random.default_rng(21).standard_normal(pr.grid.node_shape)
        for q in range(3):
            u[q][~pr.grid.dof_mask(q)] = 0.0
        u = u.astype(gp.dtype).astype(np.float64)
        _, D_ref, _, _, SD, SP = pr.residual(u, pr.grad_ustar())
        F.fftm_set_option(gp.p, F.FFTM_OPT_RESIDUAL_PASSES, 2)
        F.fftm_solve_step(gp.p)
        u_dev = torch.from_numpy(node_to_abi(u).astype(gp.dtype)).cuda()
        D_dev, norms = torch.empty_like(u_dev), torch.empty(3, dtype=torch.float64, device="cuda")
        F.fftm_residual_noalloc(gp.p, u_dev, D_dev, norms)
        torch.cuda.synchronize()
        D = node_from_abi(D_dev.cpu().numpy()).astype(np.float64)
        nm = norms.cpu().numpy()
    finally:
        gp.close()
    tol = TOL[precision]
    assert rel_l2(D, D_ref) < tol
    assert abs(nm[0] - SD) <= 10 * tol * SD and abs(nm[1] - SP) <= tol * SP
