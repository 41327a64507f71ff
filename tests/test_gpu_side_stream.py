"""Calls on a stream that does not synchronise with the default stream, with long work queued on the
default stream and none of the library's buffers made yet, against the same calls on an idle GPU: new
buffers are cleared before the caller's launches read them, and nothing waits for the default stream's
work.  The same kernels in the same order: equal bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mlmc():
    from paper_1505_00965_gb300 import build

    build.build()
    from paper_1505_00965_gb300 import mlmc as binding

    return binding


def _calls(mlmc):
    import torch

    rng = np.random.default_rng(5)
    theta = (0.2 * rng.standard_normal(mlmc.MLMC_CV_PARAMS)).astype(np.float32)
    X = torch.tensor(rng.standard_normal((4096, 16)).astype(np.float32), device="cuda")
    Y = torch.tensor(rng.standard_normal(4096).astype(np.float32), device="cuda")
    G = torch.zeros(4096, device="cuda")
    p = mlmc.Problem(payoff="asian")

    def forward(stream):
        mlmc.mlmc_mlp_forward(theta, X, 4096, G, stream=stream)
        with torch.cuda.stream(stream):
            return G.cpu().numpy()

    def estimate(mode):
        def call(stream):
            before = mlmc.mlmc_set_driver_mode(mode)
            try:
                return np.array(mlmc.mlmc_estimate(1e-2, p, 3, stream=stream).sums)
            finally:
                mlmc.mlmc_set_driver_mode(before)
        return call

    return {
        "level_sums": lambda s: np.array(mlmc.mlmc_level_sums_ex(3, 4, 30_000, 0, p, 3, precision="fp64", stream=s)[0]),
        "mlp_grad": lambda s: mlmc.mlmc_mlp_grad(theta, X, Y, 4096, stream=s)[1],
        "mlp_forward": forward,
        "estimate_host": estimate("host"),
        "estimate_device": estimate("device"),
        "estimate_batch": lambda s: np.array([e.P for e in mlmc.mlmc_estimate_batch([(p, 1e-2, 3)] * 4, stream=s)]),
        "level_sums_batch": lambda s: np.array(mlmc.mlmc_level_sums_batch([(p, 3, 2, 0, 9_999)] * 3, stream=s)),
    }


@pytest.mark.parametrize("name", ["level_sums", "mlp_grad", "mlp_forward", "estimate_host", "estimate_device",
                                  "estimate_batch", "level_sums_batch"])
def test_first_call_beside_a_busy_default_stream(mlmc, name):
    import torch

    call, side = _calls(mlmc)[name], torch.cuda.Stream()
    torch.cuda.synchronize()
    want = call(side)
    # workspaces of earlier allocations leave non-zero words where new buffers may come to lie
    dirt = torch.full((1 << 24,), -1, dtype=torch.int32, device="cuda")
    del dirt
    torch.cuda.empty_cache()
    a = torch.ones(8192, 8192, device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    mlmc.mlmc_shutdown()
    for _ in range(200):  # about 0.1 s
        a @ a
    got = call(side)
    assert np.array_equal(got, want)
    torch.cuda.synchronize()
    assert np.array_equal(call(side), want)
