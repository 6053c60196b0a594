"""Tensor-core products with many tiles and many blocks per CTA at rows that are not 16-byte aligned:
more than 32 tiles per CTA (the epilogue reads where tiles go 32 at a time) with the old C added and C's
norm map written at leaf 64, and about a dozen rounded blocks per CTA at leaf 128.  Entry-wise bounds
from the rounding of the operands (u relative, and for FP16 half a unit of its smallest subnormal
below the block's exponent) and FP32 sums."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13042_gb300 as P  # noqa: E402


def _rows(m, n, g, pad):
    """A row-major view with leading dimension n + pad."""
    return torch.randn(m, n + pad, generator=g, device="cuda")[:, :n]


def _bound(A, B, u, tiny, k, split_u=None):
    a, b = A.double().abs(), B.double().abs()
    if split_u is None:
        ra, rb = u * a + tiny, u * b + tiny
        op = ra @ b + a @ rb + ra @ rb
    else:                                 # hi and lo parts; lo * lo is left out
        op = split_u * (a @ b)
    # FP32 sums of k products, each addition within 2^-22
    return op + k * 2.0 ** -22 * ((1.0 + 4.0 * u) * (a @ b))


@pytest.mark.parametrize("schedule", ["static", "dynamic"])
@pytest.mark.parametrize("cut", [0, 3])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-1.5, 0.5)])
def test_more_than_32_tiles_per_cta(alpha, beta, cut, schedule):
    leaf, m, n, k = 64, 90 * 64 - cut, 72 * 64 - cut, 70      # 6480 tiles: 42 for each of 152 CTAs
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    A, B = _rows(m, k, g, 0), _rows(k, n, g, 0)
    C0 = _rows(m, n, g, 1 if cut else 0)
    wide = torch.full((m, C0.stride(0)), 7.0, device="cuda")
    C = wide[:, :n]
    C.copy_(C0)
    nC = torch.full((90, 72), float("nan"), dtype=torch.float64, device="cuda")
    plan = P.GeneralPlan(m, k, n, leaf, P.BF16).set_schedule(schedule)
    plan.plan_multiply(P.spamm_normmap_rect(A, leaf), P.spamm_normmap_rect(B, leaf), 0.0, A, B, C,
                       alpha=alpha, beta=beta, normC=nC)
    ref = alpha * (A.double() @ B.double()) + beta * C0.double()
    bound = abs(alpha) * _bound(A, B, 2.0 ** -9, 0.0, k) + 2.0 ** -22 * ref.abs()
    assert bool(((C.double() - ref).abs() <= bound).all())
    assert bool((wide[:, n:] == 7.0).all())                   # nothing past the rows
    pad = torch.nn.functional.pad(C.double(), (0, 72 * leaf - n, 0, 90 * leaf - m))
    norms = pad.square().view(90, leaf, 72, leaf).sum((1, 3)).sqrt()
    assert bool(((nC - norms).abs() <= 1e-12 * norms).all())


@pytest.mark.parametrize("precision,u,tiny,split_u", [
    (P.FP16, 2.0 ** -11, 2.0 ** -25 * 8.0, None),            # entries below 8: exponents up to 3
    (P.BF16, 2.0 ** -9, 0.0, None),
    (P.TF32X3, 2.0 ** -11, 0.0, 3.01 * 2.0 ** -22)])         # two residues and lo * lo
@pytest.mark.parametrize("pad", [0, 1, 2])
def test_many_blocks_per_cta_unaligned(precision, u, tiny, split_u, pad):
    leaf, s = 128, 31                                         # 1922 blocks: 12 for each of 152 CTAs
    m = s * leaf - pad
    g = torch.Generator(device="cuda")
    g.manual_seed(13 + pad)
    A, B = _rows(m, m, g, pad), _rows(m, m, g, 3 * pad)
    assert float(max(A.abs().max(), B.abs().max())) < 8.0
    C = torch.full((m, m), float("nan"), device="cuda")
    plan = P.GeneralPlan(m, m, m, leaf, precision)
    plan.plan_multiply(P.spamm_normmap_rect(A, leaf), P.spamm_normmap_rect(B, leaf), 0.0, A, B, C)
    ref = A.double() @ B.double()
    assert bool(((C.double() - ref).abs() <= _bound(A, B, u, tiny, m, split_u)).all())
