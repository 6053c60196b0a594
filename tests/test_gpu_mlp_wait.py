"""The training loop's bounded wait: the self-test withholds the exchange between the CTAs of the
cluster.  The kernel must end, all weights and losses must be NaN and the time-out must be latched
(the self-test checks these and clears its word), and training afterwards must give the bits it gave
before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13042_gb300 as P  # noqa: E402
import synth  # noqa: E402
from gpu_helpers import dev, host  # noqa: E402


def _train():
    rng = np.random.default_rng(4)
    X = np.concatenate([rng.dirichlet(np.full(64, 0.2), size=300),
                        rng.uniform(-7.0, -1.0, size=(300, 1))], axis=1).astype(np.float32)
    W = dev(synth.mlp_init(6))
    M, V = torch.zeros_like(W), torch.zeros_like(W)
    idx = rng.permutation(300)[:256].astype(np.int32).repeat(2)
    loss = P.spamm_mlp_train(W, M, V, 0, dev(X), dev(rng.normal(-6.0, 1.0, 300).astype(np.float32)),
                             dev(idx), 4, 128, 1e-3, 0.2)
    return [host(t) for t in (W, M, V, loss)]


@pytest.mark.parametrize("limit_ns", [1_000, 1_000_000])
def test_withheld_exchange_times_out(limit_ns):
    before = _train()
    assert P.spamm_last_device_status() == 0
    elapsed = P.spamm_selftest_bounded_wait(limit_ns)      # raises unless every wait gave up
    assert limit_ns <= elapsed < 1_000_000_000
    assert P.spamm_last_device_status() == 5               # the other two waits' word
    assert P.spamm_last_device_status() == 0
    for x, y in zip(before, _train()):
        assert np.array_equal(x, y)
    assert P.spamm_last_device_status() == 0
