"""Launches of few, long FP32 paths (increments formed by the block's other warps) against the plain
kernels, which an explicit samples_per_thread = 1 selects: every sample's Y bit for bit (the same
operations in the same order).  A relay thread has one sample at most, whose FP32 powers enter the FP64
sums unbatched: the four sums are those of the samples' FP32 powers, to 1e-12.  (A plain thread may
batch two in FP32: the ranges below cross a 2^32 boundary of the sample index.)"""
import numpy as np
import pytest

from gpu_helpers import run_level

pytestmark = pytest.mark.gpu

# (M, level, lanes, samples): one and several lane warps, ragged last warps, lanes of 64 calls up to
# whole paths long enough for the Asian's two-level sums, coarse steps of 2, 4 and 8
SHAPES = [(4, 4, 1, 1), (4, 5, 4, 37), (4, 6, 1, 9000), (4, 7, 16, 65), (4, 8, 32, 33), (4, 8, 16, 1003), (4, 8, 1, 3),
          (2, 9, 1, 70), (2, 13, 8, 41), (8, 4, 8, 19), (8, 3, 1, 33)]


@pytest.fixture(scope="module")
def mlmc():
    from paper_1505_00965_gb300 import build

    build.build()
    from paper_1505_00965_gb300 import mlmc as binding

    return binding


@pytest.mark.parametrize("payoff", ["european", "asian", "lookback", "digital"])
@pytest.mark.parametrize("scheme,estimator", [("em", "coupled"), ("em", "single"), ("milstein", "coupled")])
@pytest.mark.parametrize("M,level,lanes,N", SHAPES)
def test_relay_equals_plain(mlmc, M, level, lanes, N, scheme, estimator, payoff):
    for sigma in (0.2, 3.0):  # with sigma = 3 split lookback chunks may start below zero
        p = mlmc.Problem(S0=100.0, r=0.05, sigma=sigma, T=1.0, K=95.0, cash=1.0, payoff=payoff, scheme=scheme,
                         estimator=estimator)
        first = 2 ** 32 - 20
        s2, y2 = run_level(mlmc, level, M, N, first, p, 3, "fp32", launch={"lanes_per_path": lanes})
        _, y1 = run_level(mlmc, level, M, N, first, p, 3, "fp32",
                           launch={"lanes_per_path": lanes, "samples_per_thread": 1})
        assert np.array_equal(y1, y2)
        f = y2.astype(np.float32)
        powers = (f, f * f, (f * f) * f, (f * f) * (f * f))
        for k in range(4):
            w = powers[k].astype(np.float64)
            assert abs(s2[k] - w.sum()) <= 1e-12 * np.abs(w).sum()
