"""FP64 paths whose steps run in fixed point, and those just beyond the rule that chooses it, against
the oracle sample by sample.

The rule (csrc/api.cu) takes its unit from dmax = |r| h + 7 sigma sqrt(h) (Milstein: and 49 c2): the
cases below reach each of the units 2^-63 .. 2^-60 and the FP64 steps beyond, at one and several
Philox blocks per path, for every payoff with a fixed-point form, both schemes and M = 2, 4, 8.

Bound per sample: 8 (u sqrt(n + 1) + e_z max(1, sigma sqrt(T))) times the largest value of the
sample's two paths (u = 2^-53, e_z = 1e-15: the normals enter the path scaled by sigma sqrt(h), and
n of them add up like a random walk to sigma sqrt(T)).
"""
import math

import numpy as np
import pytest

import oracle

from gpu_helpers import oracle_problem, run_level

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mlmc():
    from paper_1505_00965_gb300 import build

    build.build()
    from paper_1505_00965_gb300 import mlmc as binding

    return binding


@pytest.mark.parametrize("precision", ["fp64", "fp64_stream32"])
@pytest.mark.parametrize("scheme", ["em", "milstein"])
@pytest.mark.parametrize("M,level,lanes", [(4, 1, 1), (4, 3, 1), (4, 4, 8), (2, 2, 1), (2, 6, 4), (8, 2, 1), (8, 2, 8)])
@pytest.mark.parametrize("dmax", [0.02, 0.17, 0.3, 0.48, 0.71, 0.9])
def test_units_match_oracle(mlmc, M, level, lanes, dmax, scheme, precision):
    n, N, first, seed = M ** level, 70, 2 ** 32 - 30, 11
    sigma = (dmax - 0.03 / n) * math.sqrt(n) / 7.0
    stream = "fp32" if precision == "fp64_stream32" else "fp64"
    for payoff in ("european", "asian", "lookback", "digital"):
        p = mlmc.Problem(S0=100.0, r=0.03, sigma=sigma, T=1.0, K=95.0, cash=1.0, payoff=payoff, scheme=scheme)
        op = oracle_problem(oracle, p)
        _, y = run_level(mlmc, level, M, N, first, p, seed, precision, launch={"lanes_per_path": lanes})
        for i in range(N):
            yo = oracle.level_samples(level, M, 1, op, seed=seed, first=first + i, stream=stream)[0]
            _, f, c = oracle.sample_paths(level, M, first + i, op, seed=seed, stream=stream)
            top = max(np.abs(f).max(), np.abs(c).max())
            assert abs(y[i] - yo) <= 8.0 * (2.0 ** -53 * math.sqrt(n + 1) + 1e-15 * max(1.0, sigma)) * top
