"""The rule that gives few samples of deep FP64 Milstein levels the library's form, from both sides: one call
of the least number of samples in fixed point against the same samples in halves, which take the
library's.  1e-9 of the four sums' norm, the agreement that the rule is there to keep."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mlmc():
    from paper_1505_00965_gb300 import build

    build.build()
    from paper_1505_00965_gb300 import mlmc as binding

    return binding


@pytest.mark.parametrize("precision", ["fp64", "fp64_stream32"])
@pytest.mark.parametrize("estimator", ["coupled", "antithetic"])
@pytest.mark.parametrize("M,level,N", [(2, 10, 64), (4, 5, 64), (2, 11, 4096), (2, 13, 4096), (4, 6, 4096), (4, 7, 4096)])
def test_least_samples_against_their_halves(mlmc, M, level, N, estimator, precision):
    first = 1001
    for payoff in ("european", "asian", "lookback"):
        p = mlmc.Problem(payoff=payoff, scheme="milstein", estimator=estimator)

        def sums(a, n):
            return np.array(mlmc.mlmc_level_sums_ex(level, M, n, first + a, p, 17, precision=precision)[0])

        whole, halves = sums(0, N), sums(0, N // 2) + sums(N // 2, N // 2)
        assert not np.array_equal(whole, halves)
        assert np.linalg.norm(whole - halves) <= 1e-9 * np.linalg.norm(halves)
