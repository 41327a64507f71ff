"""FP64 sums of options whose size is near the ends of the FP64 range: finite and exact to rounding.

Scaling S0, K and the sums' powers by 2^k is exact while nothing overflows or underflows, so the sums
of a scaled option are those of the plain one times 2^(k j), to a few roundings per sample: each of
the fourth powers rounds at most ten times, 1e-14 relative for sums of one sign; the sums of Y itself
cancel by less than a hundred.  Bound: 1e-12.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [("fp64", "em", 0.2), ("fp64_stream32", "em", 0.2), ("fp64", "milstein", 0.2), ("fp64", "em", 3.0)]


@pytest.fixture(scope="module")
def mlmc():
    from paper_1505_00965_gb300 import build

    build.build()
    from paper_1505_00965_gb300 import mlmc as binding

    return binding


def _sums(mlmc, level, S0, K, precision, scheme, sigma, payoff, estimator="coupled", N=1000):
    p = mlmc.Problem(S0=S0, K=K, r=0.05, sigma=sigma, T=1.0, payoff=payoff, scheme=scheme, estimator=estimator)
    return np.array(mlmc.mlmc_level_sums_ex(level, 4, N, 5, p, 3, precision=precision)[0])


# 2^250: disc S0 to the fourth power overflows, the sums do not (differences of levels 1 and 2 only)
@pytest.mark.parametrize("k,levels", [(250, (1, 2)), (-1000, (0, 1, 2, 3))])
@pytest.mark.parametrize("precision,scheme,sigma", CASES)
def test_sums_scale_with_the_option(mlmc, precision, scheme, sigma, k, levels):
    for payoff in ("european", "asian", "lookback"):
        for level in levels:
            if k > 0 and sigma > 1:
                continue  # the sums of fourth powers do overflow
            want = _sums(mlmc, level, 100.0, 100.0, precision, scheme, sigma, payoff)
            got = _sums(mlmc, level, math.ldexp(100.0, k), math.ldexp(100.0, k), precision, scheme, sigma, payoff)
            for j in range(1, 5 if k > 0 else 2):
                scaled = math.ldexp(math.ldexp(got[j - 1], -k * (j // 2)), -k * (j - j // 2))
                assert math.isclose(scaled, want[j - 1], rel_tol=1e-12), (payoff, level, j)
    if k > 0 or precision != "fp64":
        return
    # batched rounds take the same payoffs
    p = [mlmc.Problem(S0=s, K=s, r=0.05, sigma=sigma, T=1.0, payoff="asian") for s in (100.0, math.ldexp(100.0, k))]
    a, b = mlmc.mlmc_level_sums_batch([(q, 3, 2, 5, 1000) for q in p], precision=precision)
    assert math.isclose(math.ldexp(b[0], -k), a[0], rel_tol=1e-12)


@pytest.mark.parametrize("precision,scheme,sigma", CASES)
def test_strike_beyond_the_range_of_the_ratio(mlmc, precision, scheme, sigma):
    # K / S0 overflows; the call with a strike of -1 pays disc (S + 1) = disc
    for payoff in ("european", "asian", "lookback"):
        for level in (0, 1, 2, 4):
            s = _sums(mlmc, level, 1e-310, -1.0, precision, scheme, sigma, payoff, "single")
            assert np.allclose(s, 1000 * math.exp(-0.05) ** np.arange(1, 5), rtol=1e-12, atol=0)
            if level:
                assert not _sums(mlmc, level, 1e-310, -1.0, precision, scheme, sigma, payoff).any()
