"""FP32 multiply at the edges of its pieces: inner dimensions that end inside a 16-wide slice, rows
16-byte aligned or not (copies of 16 or of 4 bytes), tiles cut by the matrix, tiles inside it; fixed
and counter order; empty tiles written by the multiply itself."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13042_gb300 as P  # noqa: E402


@pytest.mark.parametrize("schedule", ["static", "dynamic"])
@pytest.mark.parametrize("leaf", [32, 64, 128])
@pytest.mark.parametrize("m,k,n", [(1, 1, 1), (33, 17, 65), (256, 256, 384), (130, 300, 261),
                                   (516, 132, 388)])
def test_fp32_tiles(m, k, n, leaf, schedule):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + k + n + leaf)
    A = torch.randn(m, k, generator=g, device="cuda")
    B = torch.randn(k, n, generator=g, device="cuda")
    A[: min(leaf, m // 2)] = 0.0                      # the first block row: empty tiles
    nA, nB = P.spamm_normmap_rect(A, leaf), P.spamm_normmap_rect(B, leaf)
    C = torch.full((m, n), float("nan"), device="cuda")
    plan = P.GeneralPlan(m, k, n, leaf, P.FP32).set_schedule(schedule)
    for _ in range(2):
        plan.plan_multiply(nA, nB, 1e-6, A, B, C)
        ref = A.double() @ B.double()
        # one FMA chain of k terms per entry
        bound = k * 2.0 ** -24 * 1.01 * (A.double().abs() @ B.double().abs())
        assert bool(((C.double() - ref).abs() <= bound).all())
    assert bool((C[: min(leaf, m // 2)] == 0.0).all())
