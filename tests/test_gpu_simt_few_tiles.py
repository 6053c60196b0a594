"""FP32 multiply with few tiles (four warps per tile) and with many (one or two): the same product
alone and repeated below itself until it has many tiles must give the same bits, at inner dimensions
that end inside a 16-wide and a 32-wide slice, tiles cut by the matrix, aligned and other rows, old C
added and C's norm map written, from one tile to the limits of the form."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13042_gb300 as P  # noqa: E402


def _product(A, B, C0, leaf, schedule, alpha, beta):
    m, k = A.shape
    n = B.shape[1]
    nA, nB = P.spamm_normmap_rect(A, leaf), P.spamm_normmap_rect(B, leaf)
    C = C0.clone()
    nC = torch.full((-(-m // leaf), -(-n // leaf)), float("nan"), dtype=torch.float64, device="cuda")
    plan = P.GeneralPlan(m, k, n, leaf, P.FP32).set_schedule(schedule)
    plan.plan_multiply(nA, nB, 1e-6, A, B, C, alpha=alpha, beta=beta, normC=nC)
    return C, nC


@pytest.mark.parametrize("schedule", ["static", "dynamic"])
@pytest.mark.parametrize("leaf", [32, 64])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-1.5, 0.5)])
@pytest.mark.parametrize("rows,cols,k", [(1, 1, 1), (1, 3, 2113), (2, 5, 1044), (12, 25, 300),
                                         (19, 24, 132)])
def test_few_and_many_tiles_give_the_same_bits(rows, cols, k, alpha, beta, leaf, schedule):
    ragged = 0 if (rows, cols) == (12, 25) else 1             # aligned rows: whole tiles
    m, n = rows * leaf, cols * leaf - 3 * ragged
    g = torch.Generator(device="cuda")
    g.manual_seed(rows * cols + k)
    A = torch.randn(m, k, generator=g, device="cuda")
    B = torch.randn(k, n, generator=g, device="cuda")
    if rows > 1:
        A[:leaf] = 0.0                                         # a row of empty tiles
    C0 = torch.randn(m, n, generator=g, device="cuda")
    C, nC = _product(A, B, C0, leaf, schedule, alpha, beta)
    ref = alpha * (A.double() @ B.double()) + beta * C0.double()
    # one FMA chain of k terms per entry, then the scaling by alpha and the sum
    bound = (k + 2) * 2.0 ** -24 * 1.01 * (abs(alpha) * (A.double().abs() @ B.double().abs())
                                           + abs(beta) * C0.double().abs())
    assert bool(((C.double() - ref).abs() <= bound).all())
    # copies of A below it: more than three tiles for each of 200 SMs
    copies = -(-601 // (rows * cols)) + 1
    many, n_many = _product(A.repeat(copies, 1), B, C0.repeat(copies, 1), leaf, schedule, alpha, beta)
    assert torch.equal(many, C.repeat(copies, 1))
    # the norms: sums of the same squares, merged in another order (FP64 grade)
    ok = (n_many - nC.repeat(copies, 1)).abs() <= 1e-12 * nC.repeat(copies, 1)
    assert bool(ok.all())


@pytest.mark.parametrize("schedule", ["static", "dynamic"])
@pytest.mark.parametrize("leaf", [32, 64])
@pytest.mark.parametrize("cut", [0, 3])
def test_few_tiles_among_many_empty_ones(cut, leaf, schedule):
    """Three block rows of forty hold anything: 75 tiles of 1000, the others are written as zeros."""
    m, n, k = 40 * leaf - cut, 25 * leaf - cut, 200
    g = torch.Generator(device="cuda")
    g.manual_seed(leaf + cut)
    A = torch.zeros(m, k, device="cuda")
    for i in (0, 17, 39):
        A[i * leaf:(i + 1) * leaf] = torch.randn(A[i * leaf:(i + 1) * leaf].shape, generator=g, device="cuda")
    B = torch.randn(k, n, generator=g, device="cuda")
    C, nC = _product(A, B, torch.full((m, n), float("nan"), device="cuda"), leaf, schedule, 1.0, 0.0)
    bound = k * 2.0 ** -24 * 1.01 * (A.double().abs() @ B.double().abs())     # one FMA chain per entry
    assert bool(((C.double() - A.double() @ B.double()).abs() <= bound).all())
    empty = torch.ones(40, dtype=torch.bool)
    empty[[0, 17, 39]] = False
    assert bool((nC[empty.cuda()] == 0.0).all()) and bool((nC[~empty.cuda()] > 0.0).all())
