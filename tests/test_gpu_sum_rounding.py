"""The residual's stencil sums keep a small derivative beside a large one, as the gradient's own
differences along each axis do: a displacement that falls by 1 across one voxel layer along x and
varies by b per voxel along y on one side of it, b far below the rounding of 1 (but not of itself).

With lambda = 0, mu = 1, h = 1 the shear stress 12 of the layer is b / 2 and the other stresses that
enter component 1 of D vanish, so that D_1 = -b / 2 on the nodes of the far side and 0 beyond.  Every
operation on these values is exact (powers of two and their small multiples): 4 units of rounding."""

import numpy as np
import pytest

from abi_helpers import GpuProblem, node_from_abi, node_to_abi
from paper_2607_05929_gb300 import build
from paper_2607_05929_gb300 import fftm as F
from synthetic.workloads import ISO_ELASTIC, Material, Workload, axis_bc

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    F.load_library()


@pytest.mark.parametrize("precision,b", [("fp32", 2.0 ** -32), ("fp64", 2.0 ** -62)])
@pytest.mark.parametrize("passes,tile", [(1, 8), (1, 16), (2, 0)])
def test_small_derivative_beside_a_large_one(precision, b, passes, tile):
    n = (6, 16, 9)
    wl = Workload("layer", n, np.zeros(n, dtype=np.int32), [Material(ISO_ELASTIC, (0.0, 1.0))],
                  axis_bc("N", "N", "N"), scheme="HEX1", lambda0=0.0, mu0=1.0)
    gp = GpuProblem(wl, precision, tol=1e30)
    try:
        F.fftm_set_option(gp.p, F.FFTM_OPT_RESIDUAL_PASSES, passes)
        F.fftm_set_option(gp.p, F.FFTM_OPT_RESIDUAL_TILE, tile)
        u = np.zeros((3,) + gp.N)
        u[0, 0] = b * np.arange(gp.N[1])[:, None]
        u[0, 1:] = 1.0
        gp.set_node(F.FFTM_FIELD_U, u)
        out = []
        if passes == 1:  # the problem's own field (FP32: high and low parts)
            F.fftm_apply(gp.p, F.FFTM_OP_RESIDUAL)
            out.append(gp.get_node(F.FFTM_FIELD_D))
        F.fftm_solve_step(gp.p)  # at rest at once (the tolerance): settles the form asked for
        u_dev = torch.from_numpy(node_to_abi(u).astype(gp.dtype)).cuda()
        D_dev, norms = torch.empty_like(u_dev), torch.empty(3, dtype=torch.float64, device="cuda")
        F.fftm_residual_noalloc(gp.p, u_dev, D_dev, norms)
        torch.cuda.synchronize()
        out.append(node_from_abi(D_dev.cpu().numpy()).astype(np.float64))
    finally:
        gp.close()
    unit = 2.0 ** -23 if precision == "fp32" else 2.0 ** -52
    for D in out:
        assert np.all(np.abs(D[1, 1, 1:-1, 1:-1] + 0.5 * b) <= 4 * unit * 0.5 * b)
        assert np.all(np.abs(D[1, 2:-1, 1:-1, 1:-1]) <= 4 * unit * 0.5 * b)
