"""Sums of deep FP64 Milstein levels against those recorded with the CUDA library's normals and FP64 steps.

P_l - P_{l-1} of these levels is a small difference of two paths that round at every step, so two forms of
the same path agree to 1e-9, the accuracy asked of FP64 sums, only where they round alike: 2-norm over the
four sums, as recorded (the same operations; the order of the sums gives about 1e-15 of their terms)."""
import json
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fp64_milstein_levels.json")) as f:
    CASES = json.load(f)["cases"]


@pytest.mark.parametrize("c", CASES, ids=lambda c: "M{M}l{level}-{estimator}-{payoff}-N{N}-s{seed}".format(**c))
def test_sums_as_recorded(c):
    from paper_1505_00965_gb300 import build

    build.build()
    from paper_1505_00965_gb300 import mlmc

    p = mlmc.Problem(payoff=c["payoff"], scheme=c["scheme"], estimator=c["estimator"])
    got, _ = mlmc.mlmc_level_sums_ex(c["level"], c["M"], c["N"], c["first"], p, c["seed"], precision=c["precision"])
    want = np.array([float.fromhex(v) for v in c["sums"]])
    assert np.linalg.norm(np.array(got) - want) <= 1e-9 * np.linalg.norm(want)
