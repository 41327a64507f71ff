"""The pool of call buffers between calls: bounded."""
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
