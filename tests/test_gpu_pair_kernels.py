"""Two samples per thread on packed FP32 pairs against one sample per thread: every sample's Y and the
sums bit for bit (the pairs take the same operations with the same roundings, and a thread adds its
samples in the same order), at counts around the grid's thread count."""
import numpy as np
import pytest

from gpu_helpers import run_level

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mlmc():
    from paper_1505_00965_gb300 import build

    build.build()
    from paper_1505_00965_gb300 import mlmc as binding

    return binding


@pytest.mark.parametrize("payoff", ["european", "asian", "lookback", "digital"])
@pytest.mark.parametrize("scheme,estimator", [("em", "coupled"), ("em", "single"), ("milstein", "coupled"),
                                              ("milstein", "single"), ("em", "antithetic"),
                                              ("milstein", "antithetic")])
@pytest.mark.parametrize("level", [2, 3, 5, 7])
def test_pairs_equal_singles(mlmc, level, scheme, estimator, payoff):
    p = mlmc.Problem(S0=100.0, r=0.05, sigma=0.3, T=1.5, K=95.0, cash=1.0, payoff=payoff, scheme=scheme,
                     estimator=estimator)
    shape = {"threads_per_block": 32, "blocks": 2, "lanes_per_path": 1}
    for N in (1, 64, 65, 128, 200) if level < 7 else (65,):
        first = 2 ** 32 - 70  # the range crosses a 2^32 boundary of the sample index
        s2, y2 = run_level(mlmc, level, 4, N, first, p, 5, "fp32", launch=shape)
        s1, y1 = run_level(mlmc, level, 4, N, first, p, 5, "fp32", launch=dict(shape, samples_per_thread=1))
        assert np.array_equal(y1, y2)
        assert np.array_equal(s1, s2)


@pytest.mark.parametrize("payoff", ["european", "asian", "lookback", "digital"])
@pytest.mark.parametrize("scheme,estimator", [("em", "coupled"), ("em", "single"), ("milstein", "coupled"),
                                              ("em", "antithetic"), ("milstein", "antithetic")])
def test_one_block_pairs_equal_singles(mlmc, scheme, estimator, payoff):
    """Level 1, one Philox block per sample, with and without per-sample output."""
    p = mlmc.Problem(S0=100.0, r=0.05, sigma=0.3, T=1.5, K=95.0, cash=1.0, payoff=payoff, scheme=scheme,
                     estimator=estimator)
    shape = {"threads_per_block": 32, "blocks": 2, "lanes_per_path": 1}
    for N in (1, 64, 65, 127, 128, 129, 200):
        for first in (0, 2 ** 32 - 70):
            s2, y2 = run_level(mlmc, 1, 4, N, first, p, 5, "fp32", launch=shape)
            s1, y1 = run_level(mlmc, 1, 4, N, first, p, 5, "fp32", launch=dict(shape, samples_per_thread=1))
            assert np.array_equal(y1, y2)
            assert np.array_equal(s1, s2)
            s0 = mlmc.mlmc_level_sums_ex(1, 4, N, first, p, 5, precision="fp32", launch=shape)[0]
            assert np.array_equal(np.asarray(s0), np.asarray(s1))
