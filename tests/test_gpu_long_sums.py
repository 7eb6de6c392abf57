"""Sliced products of long K with operands whose digits all have one sign: the
integer sums reach their bounds.

Every digit of x is 2^w - 1 at either width (x = sum_p (2^w - 1) 2^-w 2^(-(w + 1) p),
rounded to FP64), so a diagonal of digit pairs adds up without cancellation.
Tolerance, relative: the dropped pairs are below (D - 1) 2^-rD * 4 (see the digit
tests), D r >= 56; every range of K is rounded a few times into C: 16 eps.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,slices,k", [(8, 7, 32513), (8, 7, 300001), (8, 6, 1000000), (7, 7, 130049), (7, 7, 9000001),
                                           (7, 8, 6000001)])
def test_long_same_sign_sums(bits, slices, k):
    import paper_1911_11906_gb300 as F
    m, n = 3, 2
    top = 2.0 ** bits - 1
    x = sum(top * 2.0 ** (-bits - (bits + 1) * p) for p in range(9))
    assert 0.5 < x < 1.0
    A = torch.full((m, k), x, dtype=torch.float64, device="cuda").t()  # (k, m), contiguous along k
    A[:, 1] *= -1.0
    Bc = torch.full((n, k), x, dtype=torch.float64, device="cuda").t()
    ctx = F.Context(wait_timeout_s=5.0)
    ctx.set_schedule("ozaki_bits", bits)
    got = F.dgemm_ozaki(A, Bc, trans_a=True, slices=slices, ctx=ctx)
    ref = k * x * x  # within 2 eps
    digits = (9, min(slices, 7)) if bits == 8 else (8, 9 if slices == 8 else slices)
    r, D = digits
    tol = 4 * (D + 1) * 2.0 ** (-r * D) + 16 * torch.finfo(torch.float64).eps
    sign = torch.tensor([1.0, -1.0, 1.0], dtype=torch.float64, device="cuda")[:, None]
    assert float(((got * sign - ref).abs() / ref).max()) <= tol


def test_ranges_of_k_with_beta_and_strided_operands():
    """K past one range, op(A) strided and beta != 0: the ranges add up as one product."""
    import paper_1911_11906_gb300 as F
    m, n, k = 5, 3, 140000
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn(k, m, dtype=torch.float64, device="cuda", generator=g).t()  # (m, k), contiguous along m
    Bc = torch.randn(n, k, dtype=torch.float64, device="cuda", generator=g).t()
    C = torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()
    ref = -2.0 * (A @ Bc) + 0.5 * C
    got = F.dgemm_ozaki(A, Bc, alpha=-2.0, beta=0.5, C=C.t().clone().t(), slices=7, ctx=F.Context(wait_timeout_s=5.0))
    bound = 2.0 * (k * 4 * 8 * 2.0 ** -56 * A.abs().amax(1)[:, None] * Bc.abs().amax(0)[None, :]
                   + (k + 28) * torch.finfo(torch.float64).eps * (A.abs() @ Bc.abs()))
    assert torch.all((got - ref).abs() <= bound)
