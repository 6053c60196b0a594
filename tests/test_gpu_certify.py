"""The certified reference tau against the same bisection in FP64 on the host: norm maps of one
block, of a partial word of k, of several units and words, of decades of range, with zeros."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13042_gb300 as P  # noqa: E402


def _bisect(nA, nB, ref_rel):
    p = nA[:, :, None] * nB[None, :, :]
    ab = math.sqrt(float((nA * nA).sum())) * math.sqrt(float((nB * nB).sum()))
    lo, hi = -60.0, 0.0
    for _ in range(36):
        mid = 0.5 * (lo + hi)
        tile = np.where(p < ab * 10.0 ** mid, p, 0.0).sum(1)
        ok = math.sqrt(float((tile * tile).sum())) <= ref_rel * ab
        lo, hi = (mid, hi) if ok else (lo, mid)
    return ab * 10.0 ** lo, ab


@pytest.mark.parametrize("bd", [1, 5, 33, 47, 64])
@pytest.mark.parametrize("ref_rel", [1e-11, 1e-3])
def test_certified_tau(bd, ref_rel):
    leaf = 32
    g = np.random.default_rng(bd)
    d = np.abs(np.arange(bd)[:, None] - np.arange(bd)[None, :])
    maps = [np.exp2(-1.7 * d) * g.uniform(0.5, 1.0, size=(bd, bd)) for _ in range(2)]
    maps[0][g.uniform(size=(bd, bd)) < 0.1] = 0.0
    maps[0][0, 0] = 1.0
    want, ab = _bisect(*maps, ref_rel)
    plan = P.Plan(bd * leaf, leaf, P.FP32)
    got, got_ab = plan.tau_certify(*(torch.from_numpy(x).cuda() for x in maps), ref_rel)
    assert got_ab == pytest.approx(ab, rel=1e-14)
    # the skip set changes only where a product is crossed: the grid point is the same, up to
    # products that meet it within the FP32 sums' 1e-6
    assert got == pytest.approx(want, rel=1e-5)
