"""Plan kernels at the edges of their units (32 tiles: 8 block rows x 4 block columns, fewer rows in
the last band, other splits below 8 block rows), of their 32-wide words of k and of the unit table
(more than 1024 units: totals by groups), on norm maps given directly: the queues must equal the
FP64 pair test triple by triple, zero, infinite, NaN and tying norms included."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13042_gb300 as P  # noqa: E402

SHAPES = [(1, 1, 1), (1, 33, 40), (2, 1024, 3), (3, 64, 7), (7, 31, 9), (8, 32, 4), (9, 65, 13),
          (16, 96, 5), (47, 47, 47), (190, 5, 190), (1030, 2, 9)]


def _norm_maps(bm, bk, bn, seed):
    g = np.random.default_rng(seed)
    out = []
    for shape in ((bm, bk), (bk, bn)):
        x = np.exp2(g.uniform(-60.0, 5.0, size=shape))
        x[g.uniform(size=shape) < 0.1] = 0.0
        x[g.uniform(size=shape) < 0.2] = 2.0 ** -3          # ties with tau = 2^-6
        x[g.uniform(size=shape) < 0.002] = np.inf
        x[g.uniform(size=shape) < 0.002] = np.nan
        out.append(x)
    return out


def _expected(nA, nB, tau):
    with np.errstate(invalid="ignore"):
        return ~(nA[:, :, None] * nB[None, :, :] < tau)       # [i, k, j]


@pytest.mark.parametrize("bm,bk,bn", SHAPES)
@pytest.mark.parametrize("tau", [0.0, 2.0 ** -6, np.inf])
def test_queues_equal_the_pair_test(bm, bk, bn, tau):
    leaf = 32
    nA, nB = _norm_maps(bm, bk, bn, 7 * bm + bk)
    want = _expected(nA, nB, tau)
    plan = P.GeneralPlan(bm * leaf, bk * leaf, bn * leaf, leaf, P.FP32)
    plan.plan(torch.from_numpy(nA).cuda(), torch.from_numpy(nB).cuda(), tau)
    tp, kk = plan.export()
    per_tile = want.sum(1)                                    # [bm, bn]
    assert np.array_equal(np.diff(tp), per_tile.ravel())
    listed = np.concatenate([np.broadcast_to(np.arange(bk), (bn, bk))[want[i].T] for i in range(bm)])
    assert np.array_equal(kk, listed.astype(np.uint16))
    st = plan.stats()
    assert st["survivors"] == int(want.sum())
    assert st["nonempty_tiles"] == int((per_tile > 0).sum())
    assert st["max_tile_survivors"] == int(per_tile.max())
    # skipped-product bounds: FP32 sums of at most bk terms per tile, then over the tiles
    fin = np.where(want, 0.0, nA[:, :, None] * nB[None, :, :])
    tile = fin.sum(1)
    assert st["skipped_bound1"] == pytest.approx(tile.sum(), rel=1e-5, abs=0)
    assert st["skipped_bound2"] == pytest.approx(np.sqrt((tile * tile).sum()), rel=1e-5, abs=0)


def test_grouped_totals_order_every_tile():
    """More than 1024 units: every non-empty tile is multiplied and every empty one zeroed."""
    bm, bk, bn, leaf = 190, 3, 190, 32
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    A = torch.randn(bm * leaf, bk * leaf, generator=g, device="cuda")
    B = torch.randn(bk * leaf, bn * leaf, generator=g, device="cuda")
    keep = torch.rand(bm, bk, generator=g, device="cuda") < 0.2
    A *= keep.repeat_interleave(leaf, 0).repeat_interleave(leaf, 1)
    nA, nB = P.spamm_normmap_rect(A, leaf), P.spamm_normmap_rect(B, leaf)
    C = torch.full((bm * leaf, bn * leaf), float("nan"), device="cuda")
    P.GeneralPlan(bm * leaf, bk * leaf, bn * leaf, leaf, P.FP32).plan_multiply(nA, nB, 1e-3, A, B, C)
    ref = A.double() @ B.double()
    # FP32 chains of bk * leaf FMAs
    bound = bk * leaf * 2.0 ** -24 * 1.01 * (A.double().abs() @ B.double().abs()) + 1e-30
    assert bool(((C.double() - ref).abs() <= bound).all())
