"""The plans of the FFT passes in FP32 (other tiles, pads, threads and registers than FP64) at the
lengths of the FP64 plan tests, and the periodic lengths above those, up to the longest that is taken.

Tolerances are the FP64 plan tests' in units of rounding: 90 units of the matrix norm times the input's
for one transform and its inverse twice that, 270 for three axes, 540 there and back, in FP32 units of
2^-24; the Green update as in the other FP32 tests."""

import numpy as np
import pytest

import synthetic as syn
from abi_helpers import GpuProblem, rel_l2
from oracle.bc import Grid, dof_range
from oracle.solver import Problem
from paper_2607_05929_gb300 import build
from paper_2607_05929_gb300 import fftm as F
from synthetic.workloads import ISO_ELASTIC, Material, Workload
from test_gpu_dt_plans import PAIRS, SIZES, dense, dense_3d

pytestmark = pytest.mark.gpu

LONG = [576, 648, 729, 768]  # periodic axes only
U32 = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    F.load_library()


def _problem(nn, pairs, precision):
    bc = [[[p[0]] * 3, [p[1]] * 3] for p in pairs]
    mats = [Material(ISO_ELASTIC, (1.0, 0.7)), Material(ISO_ELASTIC, (3.0, 2.0))]
    wl = Workload("plan", tuple(nn), np.asarray(syn.laminate(tuple(nn), 0, max(1, nn[0] // 2)), np.uint16), mats, bc,
                  scheme="TETRA2", lambda0=1.3, mu0=0.8)
    return wl, GpuProblem(wl, precision)


@pytest.mark.parametrize("n", LONG)
def test_long_periodic_rows_match_the_dense_sums(n):
    M = dense("DFT", n)
    x = np.random.default_rng(n).standard_normal(n)
    X = F.fftm_dt1d("DFT", n, x)
    assert np.linalg.norm(X - M @ x) <= 1e-14 * np.linalg.norm(M, 2) * np.linalg.norm(x)
    back = F.fftm_dt1d("DFT", n, X, inverse=True)
    assert np.linalg.norm(back - x) <= 2e-14 * np.linalg.norm(x)


@pytest.mark.parametrize("kind,n", [(k, n) for k in PAIRS for n in SIZES] + [("DFT", n) for n in LONG])
def test_fp32_rows_match_the_dense_sums(kind, n):
    wl, gp = _problem([n, 2, 2], [PAIRS[kind], PAIRS["DFT"], PAIRS["DFT"]], "fp32")
    M, (lo, hi) = dense(kind, n), dof_range(kind, n)
    try:
        x = np.zeros((3,) + gp.N)
        x[:, lo:hi] = np.random.default_rng(n).standard_normal((3, hi - lo, 1, 1))  # constant along y and z
        x = x.astype(np.float32).astype(np.float64)
        gp.set_node(F.FFTM_FIELD_WORK, x)
        F.fftm_apply(gp.p, F.FFTM_OP_DT_FORWARD)
        X = gp.get_node(F.FFTM_FIELD_WORK)
        F.fftm_apply(gp.p, F.FFTM_OP_DT_INVERSE)
        back = gp.get_node(F.FFTM_FIELD_WORK)
    finally:
        gp.close()
    for q in range(3):
        line = x[q, lo:hi, 0, 0]
        size = np.linalg.norm(M, 2) * np.linalg.norm(line)
        assert np.linalg.norm(X[q, lo:hi, 0, 0] / 4 - M @ line) <= 90 * U32 * size, q
        assert np.linalg.norm(back[q, lo:hi, 1, 1] - line) <= 180 * U32 * np.linalg.norm(line), q


@pytest.mark.parametrize("axis", [1, 2])
@pytest.mark.parametrize("kind,n", [(k, n) for k in PAIRS for n in (3, 8, 18, 24, 81, 108, 162, 288)] +
                         [("DFT", 576), ("DFT", 768)])
def test_fp32_pencils_and_the_fused_pass_match_the_oracle(kind, n, axis):
    nn = [36, 4, 4]  # more than one tile of 32 pencils along x, the last one ragged
    nn[axis] = n
    pairs = [PAIRS["DCT1"], PAIRS["DST1"], PAIRS["DFT"]]
    pairs[axis] = PAIRS[kind]
    wl, gp = _problem(nn, pairs, "fp32")
    g = Grid(wl.n, wl.bc)
    try:
        x = np.random.default_rng(10 * n + axis).standard_normal(g.node_shape).astype(np.float32).astype(np.float64)
        for q in range(3):
            x[q][~g.dof_mask(q)] = 0.0
        gp.set_node(F.FFTM_FIELD_WORK, x)
        F.fftm_apply(gp.p, F.FFTM_OP_DT_FORWARD)
        got = gp.get_node(F.FFTM_FIELD_WORK)
        for q in range(3):
            assert rel_l2(got[q], dense_3d(x[q], g.kind[q], g.n)) < 270 * U32, q
        F.fftm_apply(gp.p, F.FFTM_OP_DT_INVERSE)
        assert rel_l2(gp.get_node(F.FFTM_FIELD_WORK), x) < 540 * U32
        gp.set_node(F.FFTM_FIELD_WORK, x)
        F.fftm_apply(gp.p, F.FFTM_OP_GREEN_UPDATE)
        assert rel_l2(gp.get_node(F.FFTM_FIELD_U), Problem(wl).green_update(x)) < 2e-5
    finally:
        gp.close()
