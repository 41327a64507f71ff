"""The pool of call buffers between calls: bounded, and a set serves any call after any other."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mlmc():
    from paper_1505_00965_gb300 import build

    build.build()
    from paper_1505_00965_gb300 import mlmc as binding

    return binding


def test_a_large_grids_workspace_is_given_back(mlmc):
    import torch

    def call(blocks):
        return mlmc.mlmc_level_sums_ex(2, 4, 1000, 0, mlmc.Problem(), 3, precision="fp32",
                                       launch={"threads_per_block": 32, "blocks": blocks, "lanes_per_path": 1})[0]

    want = call(32)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for blocks in (1 << 21, 3 << 20):  # 64 and 96 MiB of block sums
        assert np.allclose(call(blocks), want, rtol=1e-5, atol=1e-3)
    assert torch.cuda.mem_get_info()[0] > free - (32 << 20)


def test_estimate_after_a_gradient_on_the_same_buffers(mlmc):
    """The gradient's parameters and outputs lie over the later slots' tickets of the driver's workspace."""
    import torch

    rng = np.random.default_rng(5)
    theta = (0.2 * rng.standard_normal(mlmc.MLMC_CV_PARAMS)).astype(np.float32)
    X = torch.tensor(rng.standard_normal((65536, 16)).astype(np.float32), device="cuda")
    Y = torch.tensor(rng.standard_normal(65536).astype(np.float32), device="cuda")
    before = mlmc.mlmc_set_driver_mode("host")
    try:
        mlmc.mlmc_shutdown()
        want = mlmc.mlmc_estimate(1e-2, mlmc.Problem(payoff="asian"), 3).sums
        mlmc.mlmc_shutdown()
        mlmc.mlmc_mlp_grad(theta, X, Y, 65536)
        got = mlmc.mlmc_estimate(1e-2, mlmc.Problem(payoff="asian"), 3).sums
    finally:
        mlmc.mlmc_set_driver_mode(before)
    assert np.array_equal(np.asarray(got), np.asarray(want))
