"""Gradient and training loop of the learned-tau network at the edges of their chunks (16 samples)
and of the cluster (a chunk per CTA and round): fewer samples than one chunk, one past a round, many
rounds.  Tolerances as in the existing comparison with the FP64 network."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13042_gb300 as P  # noqa: E402
import synth  # noqa: E402
from gpu_helpers import dev, host  # noqa: E402
from oracle import mlp as OM  # noqa: E402


def _samples(count, seed):
    rng = np.random.default_rng(seed)
    X = np.concatenate([rng.dirichlet(np.full(64, 0.2), size=count),
                        rng.uniform(-7.0, -1.0, size=(count, 1))], axis=1).astype(np.float32)
    return X, rng.normal(-6.0, 1.0, size=count).astype(np.float32)


@pytest.mark.parametrize("count", [1, 15, 16, 17, 127, 128, 255, 256, 257, 1000])
def test_gradient_chunk_edges(count):
    theta = synth.mlp_init(3)
    X, Y = _samples(count, count)
    g, loss = P.spamm_mlp_grad(dev(theta), dev(X), dev(Y), 0.1)
    ref_loss, ref_g = OM.loss_and_grad(theta.astype(np.float64), X.astype(np.float64),
                                       Y.astype(np.float64), 0.1)
    assert abs(float(host(loss)[0]) - ref_loss) <= 1e-5 * max(1.0, abs(ref_loss))
    assert np.max(np.abs(host(g).astype(np.float64) - ref_g)) <= 1e-4 * np.max(np.abs(ref_g))


@pytest.mark.parametrize("batch", [1, 16, 100, 256, 272, 600])
def test_training_batch_edges(batch):
    theta = synth.mlp_init(8).astype(np.float64)
    X, Y = _samples(700, 5)
    steps, lr, q = 3, 1e-3, 0.2
    rng = np.random.default_rng(batch)
    idx = np.stack([rng.permutation(700)[:batch] for _ in range(steps)]).astype(np.int32)
    W = dev(theta.astype(np.float32))
    M, V = torch.zeros_like(W), torch.zeros_like(W)
    losses = host(P.spamm_mlp_train(W, M, V, 0, dev(X), dev(Y), dev(idx.ravel()), steps, batch, lr, q))
    m, v = np.zeros_like(theta), np.zeros_like(theta)
    for s in range(steps):
        loss, g = OM.loss_and_grad(theta, X[idx[s]].astype(np.float64), Y[idx[s]].astype(np.float64), q)
        assert abs(losses[s] - loss) <= 1e-4 * max(1.0, abs(loss))
        theta, m, v = OM.adam_step(theta, g, m, v, s + 1, lr)
    assert np.max(np.abs(host(W) - theta)) <= 5e-5
