"""Queue expansion at the line between its two forms (up to 16 entries per tile of a unit on
average a lane writes a tile's entries, above it a warp), over several words of k, with split
flags, and the list of needed blocks (a block missing from it would be multiplied unrounded).

Exact: the entries are whole numbers, and the flags follow from one FP64 product each."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13042_gb300 as P  # noqa: E402


@pytest.mark.parametrize("bm,bk,bn", [(8, 15, 4), (8, 16, 4), (8, 17, 4), (9, 33, 5), (3, 130, 11),
                                      (40, 140, 40), (24, 1024, 8)])
@pytest.mark.parametrize("keep", [1.0, 0.12, 16.0])
def test_entries_and_flags(bm, bk, bn, keep):
    """keep: the fraction of the triples that survive (16: about 16 per tile)."""
    leaf = 64
    g = np.random.default_rng(bm * bk + bn)
    nA, nB = np.exp2(g.uniform(-40, 0, (bm, bk))), np.exp2(g.uniform(-40, 0, (bk, bn)))
    p = nA[:, :, None] * nB[None, :, :]
    frac = min(1.0, keep / bk if keep > 1 else keep)
    tau = 0.0 if frac == 1.0 else float(np.quantile(p, 1.0 - frac))
    want = ~(p < tau)
    plan = P.GeneralPlan(bm * leaf, bk * leaf, bn * leaf, leaf, P.BF16_SPLIT)
    plan.plan(torch.from_numpy(nA).cuda(), torch.from_numpy(nB).cuda(), tau, target_rel_err=1e-6)
    tp, kk = plan.export()
    st = plan.stats()
    assert np.array_equal(np.diff(tp), want.sum(1).ravel())
    ijk = np.argwhere(want.transpose(0, 2, 1))              # (i, j, k) in queue order
    assert np.array_equal(kk & 0x3FF, ijk[:, 2].astype(np.uint16))
    inv = 1.0 / (st["norm_a"] * st["norm_b"])
    rel = p.transpose(0, 2, 1)[want.transpose(0, 2, 1)] * inv
    binade = np.clip(np.floor(np.log2(rel)), -200, 1)
    clear = np.abs(np.log2(rel) - np.round(np.log2(rel))) > 1e-9   # log2 itself is rounded
    flags = (kk & 0x8000) != 0
    assert np.array_equal(flags[clear], (binade >= st["flag_exponent"])[clear])
    assert int(flags.sum()) == st["flagged"]


@pytest.mark.parametrize("bk", [5, 33])
def test_every_needed_block_is_rounded(bk):
    """A product whose survivors use a few scattered blocks equals the sum over them: FP32 sums
    of FP16 products, exact here (small whole numbers)."""
    bm, bn, leaf = 19, 11, 64
    g = torch.Generator(device="cuda").manual_seed(bk)
    A = torch.randint(-3, 4, (bm * leaf, bk * leaf), device="cuda", generator=g).float()
    B = torch.randint(-3, 4, (bk * leaf, bn * leaf), device="cuda", generator=g).float()
    keep = torch.rand(bm, bk, device="cuda", generator=g) < 0.15
    A *= keep.repeat_interleave(leaf, 0).repeat_interleave(leaf, 1)
    nA, nB = P.spamm_normmap_rect(A, leaf), P.spamm_normmap_rect(B, leaf)
    C = torch.full((bm * leaf, bn * leaf), float("nan"), device="cuda")
    plan = P.GeneralPlan(bm * leaf, bk * leaf, bn * leaf, leaf, P.FP16)
    for _ in range(2):
        plan.plan_multiply(nA, nB, 1.0, A, B, C)
        assert torch.equal(C, (A.double() @ B.double()).float())
