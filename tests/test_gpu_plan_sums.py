"""Sums of skipped products: a large term among small ones, each of which a plain FP32 chain would
lose.  The bounds are derived from the roundings a term meets."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13042_gb300 as P  # noqa: E402

# two norms and their product rounded to FP32, three pairwise additions of a group of eight,
# the compensated running sum and its compensation, two pairwise additions of the warps'
# shares: 10 roundings of at most 2^-24 each; one more for the square root's argument
SUM_REL = 11 * 2.0 ** -24


@pytest.mark.parametrize("spread", [0, 1, 40])
@pytest.mark.parametrize("bk", [8, 31, 64, 257, 1024])
def test_skipped_sums_keep_small_terms(bk, spread):
    """One tile: one product of 1, the others about 2^-25 (or, with a spread, falling by half every
    `spread` of k), all of them skipped."""
    leaf = 32
    p = np.full(bk, 2.0 ** -25)
    if spread:
        p *= 2.0 ** -(np.arange(bk) // spread % 60).astype(np.float64)
    p[bk // 3] = 1.0
    plan = P.GeneralPlan(leaf, bk * leaf, leaf, leaf, P.FP32)
    plan.plan(torch.from_numpy(p[None, :]).cuda(), torch.ones(bk, 1, dtype=torch.float64, device="cuda"), 2.0)
    st = plan.stats()
    assert st["survivors"] == 0
    assert abs(st["skipped_bound1"] - p.sum()) <= SUM_REL * p.sum()
    assert abs(st["skipped_bound2"] - p.sum()) <= SUM_REL * p.sum()


def test_certified_tau_counts_small_terms():
    """The bound is admissible without the small products and not with them: the certified tau must
    not pass the large product."""
    bd, leaf = 256, 32
    p = np.full(bd, 2.0 ** -26)
    p[0], p[100] = 0.5, 1.0
    small = (bd - 2) * 2.0 ** -26
    nA, nB = np.zeros((bd, bd)), np.zeros((bd, bd))
    nA[0], nB[:, 0] = p, 1.0
    ab = float(np.sqrt((p * p).sum()) * np.sqrt(bd))
    # between the true sum 0.5 + small and the sum without a tenth of the small products: a chain
    # over a quarter of k loses all of its share (each a quarter of the last place of 0.5)
    limit = 0.5 + 0.9 * small
    plan = P.Plan(bd * leaf, leaf, P.FP32)
    tau, norm_ab = plan.tau_certify(torch.from_numpy(nA).cuda(), torch.from_numpy(nB).cuda(), limit / ab)
    assert norm_ab == pytest.approx(ab, rel=1e-12)
    assert tau <= 0.5 * (1.0 + 1e-12)
    assert tau >= 0.5 * (1.0 - 1e-8)          # the grid's step is 10^(60 / 2^36)
