"""Every shape of the FFT passes' plans against the oracle's dense sums, in FP64: no split, one
split and two of the type-I transforms, each stage radix (2, 3, 4, 6, 8, 9, 12, 16), one to three
stages, on each axis (rows, pencils, the fused z pass), the shortest and longest lengths included.

Tolerance: an FFT of up to three stages of radix at most 16 rounds a result a few times per stage,
a handful of units of 2^-53 = 1.1e-16 relative to the norm of the matrix times the norm of the
input; 1e-14 is 90 units, against about log2(1024) = 10 one-unit steps.  The fused Green update goes through six such passes and
scales each mode by its own factor: 1e-12."""

import numpy as np
import pytest

import synthetic as syn
from abi_helpers import GpuProblem, rel_l2
from oracle.bc import Grid, dof_range
from oracle.solver import Problem
from paper_2607_05929_gb300 import build
from paper_2607_05929_gb300 import fftm as F
from synthetic.workloads import ISO_ELASTIC, Material, Workload

pytestmark = pytest.mark.gpu

SIZES = [2, 3, 4, 8, 12, 18, 24, 27, 32, 54, 72, 81, 108, 128, 162, 216, 243, 288, 432, 486, 512]
PAIRS = {"DFT": ("P", "P"), "DCT1": ("N", "N"), "DCT3": ("N", "D"), "DST1": ("D", "D"), "DST3": ("D", "N")}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    F.load_library()


def dense(kind, n):
    """The Table 1 sums (the DFT in halfcomplex order) with the angles reduced to one period in
    integers, so that the entries are good to a unit: angles of up to n pi rounded first would be
    off by n units."""
    lo, hi = dof_range(kind, n)
    j, k = np.arange(lo, hi), np.arange(hi - lo)

    def angle(num, den):  # pi num / den, num reduced modulo 2 den
        return np.pi * (num % (2 * den)) / den

    if kind == "DFT":
        a = angle(2 * np.outer(np.minimum(k, n - k), j), n)
        return np.where((2 * k <= n)[:, None], np.cos(a), -np.sin(a))
    if kind in ("DCT1", "DST1"):
        a = angle(np.outer(k if kind == "DCT1" else k + 1, j), n)
    else:
        a = angle(np.outer(2 * k + 1, j), 2 * n)
    w = np.full(j.size, 2.0)
    if kind in ("DCT1", "DCT3"):
        w[0] = 1.0
    if kind in ("DCT1", "DST3"):
        w[-1] = 1.0
    return w * (np.cos(a) if kind in ("DCT1", "DCT3") else np.sin(a))


def dense_3d(x, kinds, n):
    s = tuple(slice(*dof_range(kinds[a], n[a])) for a in range(3))
    y = x[s]
    for a in range(3):
        y = np.moveaxis(np.moveaxis(y, a, -1) @ dense(kinds[a], n[a]).T, -1, a)
    out = np.zeros_like(x)
    out[s] = y
    return out


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", list(PAIRS))
def test_rows_match_the_dense_sums(kind, n):
    M = dense(kind, n)
    x = np.random.default_rng(n).standard_normal(M.shape[0])
    X = F.fftm_dt1d(kind, n, x)
    ref = M @ x
    assert np.linalg.norm(X - ref) <= 1e-14 * np.linalg.norm(M, 2) * np.linalg.norm(x)
    back = F.fftm_dt1d(kind, n, X, inverse=True)
    assert np.linalg.norm(back - x) <= 2e-14 * np.linalg.norm(x)


@pytest.mark.parametrize("axis", [1, 2])
@pytest.mark.parametrize("n", [3, 8, 18, 24, 81, 108, 162, 288])
@pytest.mark.parametrize("kind", list(PAIRS))
def test_pencils_and_the_fused_pass_match_the_oracle(kind, n, axis):
    nn = [36, 4, 4]  # more than one tile of 16 pencils along x, the last one ragged
    nn[axis] = n
    pairs = [PAIRS["DCT1"], PAIRS["DST1"], PAIRS["DFT"]]
    pairs[axis] = PAIRS[kind]
    bc = [[[p[0]] * 3, [p[1]] * 3] for p in pairs]
    phase = syn.laminate(tuple(nn), 0, 6)
    mats = [Material(ISO_ELASTIC, (1.0, 0.7)), Material(ISO_ELASTIC, (3.0, 2.0))]
    wl = Workload("plan", tuple(nn), np.asarray(phase, np.uint16), mats, bc, scheme="TETRA2", lambda0=1.3, mu0=0.8)
    g = Grid(wl.n, wl.bc)
    gp = GpuProblem(wl, "fp64")
    try:
        x = np.random.default_rng(10 * n + axis).standard_normal(g.node_shape)
        for q in range(3):
            x[q][~g.dof_mask(q)] = 0.0
        gp.set_node(F.FFTM_FIELD_WORK, x)
        F.fftm_apply(gp.p, F.FFTM_OP_DT_FORWARD)
        got = gp.get_node(F.FFTM_FIELD_WORK)
        for q in range(3):
            assert rel_l2(got[q], dense_3d(x[q], g.kind[q], g.n)) < 3e-14, q
        F.fftm_apply(gp.p, F.FFTM_OP_DT_INVERSE)
        assert rel_l2(gp.get_node(F.FFTM_FIELD_WORK), x) < 6e-14
        gp.set_node(F.FFTM_FIELD_WORK, x)
        F.fftm_apply(gp.p, F.FFTM_OP_GREEN_UPDATE)
        assert rel_l2(gp.get_node(F.FFTM_FIELD_U), Problem(wl).green_update(x)) < 1e-12
    finally:
        gp.close()


def test_dismissed_nodes_stay_zero():
    """Components with different conditions on one axis: the nodes that a component does not transform
    (its Dirichlet nodes) hold exact zeros after a Green update, FP32 and FP64."""
    bc = [[["D" if q == a else "N" for q in range(3)] for _ in range(2)] for a in range(3)]
    wl = Workload("dismissed", (24, 18, 16), np.zeros((24, 18, 16), np.uint16), [Material(ISO_ELASTIC, (1.0, 0.7))], bc,
                  scheme="TETRA2", lambda0=1.3, mu0=0.8)
    g = Grid(wl.n, wl.bc)
    x = np.random.default_rng(3).standard_normal(g.node_shape)
    for q in range(3):
        x[q][~g.dof_mask(q)] = 0.0
    ref = Problem(wl).green_update(x)
    for precision, tol in (("fp64", 1e-12), ("fp32", 2e-5)):
        gp = GpuProblem(wl, precision)
        try:
            gp.set_node(F.FFTM_FIELD_WORK, x)
            F.fftm_apply(gp.p, F.FFTM_OP_GREEN_UPDATE)
            u = gp.get_node(F.FFTM_FIELD_U)
            for q in range(3):
                assert not u[q][~g.dof_mask(q)].any(), (precision, q)
            assert rel_l2(u, ref) < tol
        finally:
            gp.close()
