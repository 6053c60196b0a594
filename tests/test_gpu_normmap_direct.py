"""The norm map of small operands (a CTA per 128 columns of a strip) against the pipeline that
larger operands take.

Both sum the same groups of entries in the same order, so the norms are equal bit for bit: a
small operand is compared with the same block rows inside a larger one (same columns, leading
dimension and alignment), and a small batch, whose aligned and other instances share one
launch, with the single calls.  Oracle tolerance: 3e-13 relative, the norm map's bound.
"""
import numpy as np
import pytest
import torch

import paper_2103_13042_gb300 as P
from oracle import spamm as S
from tests.gpu_helpers import dev, host

pytestmark = pytest.mark.gpu

LIMIT = 5 << 20     # entries of a launch that takes the direct kernel


@pytest.mark.parametrize("leaf", [32, 64, 128])
@pytest.mark.parametrize("rows,cols", [(1, 1), (31, 5), (64, 127), (129, 128), (200, 1030),
                                       (257, 2049), (130, 3500)])
def test_small_equals_large(rows, cols, leaf):
    """(cols % 4 decides between 16-byte and scalar reads, cols > 1024 takes several windows.)"""
    big = (LIMIT // cols // leaf + 1) * leaf
    g = torch.Generator(device="cuda").manual_seed(rows * 7 + cols)
    X = torch.randn(big, cols, device="cuda", generator=g)
    X *= 10.0 ** torch.randint(-25, 18, (big, cols), device="cuda", generator=g)
    X[:: 3, : min(cols, 40)] = 0.0
    assert big * cols > LIMIT and rows * cols <= LIMIT
    full = rows // leaf * leaf                # whole block rows: the same entries in both
    small = host(P.spamm_normmap_rect(X[:rows], leaf))
    large = host(P.spamm_normmap_rect(X, leaf))
    assert np.array_equal(small[: full // leaf], large[: full // leaf])
    if rows % leaf:                           # the ragged last block row: zeros below it
        Y = X.clone()
        Y[rows:] = 0.0
        assert np.array_equal(small, host(P.spamm_normmap_rect(Y, leaf))[: small.shape[0]])
    assert P.spamm_last_device_status() == 0


@pytest.mark.parametrize("leaf", [32, 64, 128])
def test_special_values(leaf):
    n = 150
    x = np.random.default_rng(leaf).standard_normal((n, n)).astype(np.float32)
    x[3, 7] = np.nan
    x[n - 1, n - 1] = np.inf
    x[:32, 64:] = 0.0
    x[40, 20] = np.finfo(np.float32).max
    x[70, 100] = np.float32(1e-45)
    X = dev(x)
    big = torch.zeros((LIMIT // n // leaf + 2) * leaf, n, device="cuda")
    big[:n] = X
    got = host(P.spamm_normmap_rect(X, leaf))
    assert np.array_equal(got, host(P.spamm_normmap_rect(big, leaf))[: got.shape[0]], equal_nan=True)


@pytest.mark.parametrize("leaf", [32, 64])
def test_mixed_batch_equals_single(leaf):
    """40 instances (more than a warp searches at once), aligned and not, in one launch."""
    rng = np.random.default_rng(leaf)
    ns = [int(x) for x in rng.integers(1, 330, 40)]
    As = [dev(rng.standard_normal((n, n)).astype(np.float32)) for n in ns]
    Bs = [dev(rng.standard_normal((n, n)).astype(np.float32)) for n in ns]
    Cs = [torch.empty_like(a) for a in As]
    assert 2 * sum(n * n for n in ns) <= LIMIT and len({n % 4 == 0 for n in ns}) == 2
    batch = P.Batch(ns, leaf, P.FP32, graph=False)
    batch.run(As, Bs, Cs, [0.0] * len(ns))
    for i in range(len(ns)):
        nA, nB = batch.export(i)[:2]
        for got, X in ((nA, As[i]), (nB, Bs[i])):
            assert np.array_equal(got, host(P.spamm_normmap(X, leaf)))
            assert np.allclose(got, S.normmap(host(X), leaf), rtol=3e-13, atol=0)
    batch.close()
