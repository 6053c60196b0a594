"""Adam with an infinite rate: inf * 0 is NaN for weights without a gradient, as the formula has it, in
the single step and in the training loop (the update keeps zero moments out of its divisions)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13042_gb300 as P  # noqa: E402


@pytest.mark.parametrize("loop", [False, True])
def test_infinite_rate(loop):
    W = torch.full((8449,), 0.5, device="cuda")
    M, V = torch.zeros_like(W), torch.zeros_like(W)
    if loop:
        X, Y = torch.zeros(16, 65, device="cuda"), torch.ones(16, device="cuda")
        idx = torch.arange(16, dtype=torch.int32, device="cuda")
        P.spamm_mlp_train(W, M, V, 0, X, Y, idx, 1, 16, float("inf"), 0.5)
    else:
        P.spamm_mlp_adam(W, torch.zeros_like(W), M, V, 1, float("inf"))
    assert bool(W[: 64 * 65].isnan().all())            # W1: no gradient (all features zero)
    assert bool((M[: 64 * 65] == 0).all())
