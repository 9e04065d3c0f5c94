"""The rounding of the transforms themselves: their distance from the exact sums, which sees what the
plan tests' tolerances leave room for (angles of the tables rounded before the cosine).

FP64: an FFT of N points with tables good to a unit rounds by about 0.6 u sqrt(log2 N) relative to
its result, u = 2^-53 (Schatzman 1996, the average case); the pre- and post-processing add about one
such step to the log2 N, and the bound is u sqrt(log2 N), five thirds of the average.  The sums are
formed in long double from angles reduced in integers.

FP32: roundings are unbiased, a constant that is off its FP32 value is not: it scales what it
multiplies.  Of a DFT of 256 points (two stages of radix 16) the spectrum's mean scale must not be off
by more than sqrt(1/2) alone explains, 1.7e-8 from its FP32 value on a quarter of the elements of each
stage: 0.85e-8; the 225 table entries, rounded independently, add 3e-8 / 15 = 2e-9, and the average
over 49152 outputs leaves 6e-10 of their roundings (one standard deviation each).  The bound, 2e-8, is
that plus five times both deviations."""

import numpy as np
import pytest

from abi_helpers import GpuProblem, oracle_r2r_forward
from oracle.bc import dof_range
from paper_2607_05929_gb300 import build
from paper_2607_05929_gb300 import fftm as F
from synthetic.workloads import ISO_ELASTIC, Material, Workload, axis_bc

pytestmark = pytest.mark.gpu

LD = np.longdouble
PI = 4 * np.arctan(LD(1))


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    F.load_library()


def dense(kind, n):
    lo, hi = dof_range(kind, n)
    j, k = np.arange(lo, hi), np.arange(hi - lo)

    def angle(num, den):
        return PI * (num % (2 * den)).astype(LD) / LD(den)

    if kind == "DFT":
        a = angle(2 * np.outer(np.minimum(k, n - k), j), n)
        return np.where((2 * k <= n)[:, None], np.cos(a), -np.sin(a))
    a = angle(np.outer(2 * k + 1, j), 2 * n)  # DCT3, DST3
    w = np.full(j.size, LD(2))
    w[0 if kind == "DCT3" else -1] = 1
    return w * (np.cos(a) if kind == "DCT3" else np.sin(a))


@pytest.mark.parametrize("n", [24, 81, 216, 243, 432])
@pytest.mark.parametrize("kind", ["DFT", "DCT3", "DST3"])
def test_fp64_transforms_round_like_an_fft_with_exact_tables(kind, n):
    M = dense(kind, n)
    rng = np.random.default_rng(n)
    err = {"forward": [0.0, 0.0], "inverse": [0.0, 0.0]}
    for _ in range(24):
        x = rng.standard_normal(M.shape[0])
        X = M @ x.astype(LD)
        spec = X.astype(np.float64)
        back = x.astype(LD)  # of the exact spectrum; its rounding to FP64 adds half a unit an entry
        for name, got, ref in (("forward", F.fftm_dt1d(kind, n, x), X),
                               ("inverse", F.fftm_dt1d(kind, n, spec, inverse=True), back)):
            d = got.astype(LD) - ref
            err[name][0] += float(d @ d)
            err[name][1] += float(ref @ ref)
    bound = 2.0 ** -53 * np.sqrt(np.log2(n))
    for name, (e2, r2) in err.items():
        assert np.sqrt(e2 / r2) <= bound, (name, np.sqrt(e2 / r2), bound)


def test_fp32_radix_16_stages_do_not_scale_the_spectrum():
    n = (256, 2, 2)
    wl = Workload("dft", n, np.zeros(n, dtype=np.int32), [Material(ISO_ELASTIC, (1.0, 1.0))],
                  axis_bc("P", "P", "P"), scheme="HEX1", lambda0=1.0, mu0=1.0)
    gp = GpuProblem(wl, "fp32")
    num = den = 0.0
    try:
        for seed in range(16):
            x = np.random.default_rng(seed).standard_normal((3,) + n).astype(np.float32).astype(np.float64)
            gp.set_node(F.FFTM_FIELD_WORK, x)
            F.fftm_apply(gp.p, F.FFTM_OP_DT_FORWARD)
            X = gp.get_node(F.FFTM_FIELD_WORK)
            for q in range(3):
                ref = oracle_r2r_forward(x[q], ["DFT"] * 3, n, n)
                num += float(np.vdot(X[q] - ref, ref))
                den += float(np.vdot(ref, ref))
    finally:
        gp.close()
    assert abs(num / den) <= 2e-8, num / den
