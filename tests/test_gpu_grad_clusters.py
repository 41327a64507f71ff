"""mlmc_mlp_grad on batches whose 16-row tiles do not divide over the CTAs of its clusters, against
the oracle's chain rule (bounds of test_gpu_cv.test_mlp_grad_matches_oracle: bfloat16 operands)."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1024 + 32, 16 * 8 * 16 * 3 - 32, 16 * 8 * 16 * 5 + 32, 65536 - 32])
def test_ragged_tiles(B):
    import torch

    from paper_1505_00965_gb300 import build

    build.build()
    from paper_1505_00965_gb300 import mlmc

    rng = np.random.default_rng(B)
    X = rng.standard_normal((B, omlp.D)).astype(np.float32)
    Y = (np.sin(X[:, 0]) + 0.5 * X[:, 1] * X[:, 2]).astype(np.float32)
    theta = omlp.init_params(3).astype(np.float32)
    loss, grad = mlmc.mlmc_mlp_grad(theta, torch.tensor(X, device="cuda"), torch.tensor(Y, device="cuda"), B)
    want_loss, want = omlp.loss_and_grad(theta.astype(np.float64), X.astype(np.float64), Y.astype(np.float64),
                                         quantize=True)
    assert abs(loss - want_loss) <= 1e-2 * want_loss
    assert np.linalg.norm(grad.astype(np.float64) - want) <= 2e-2 * np.linalg.norm(want)
