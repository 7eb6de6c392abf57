"""FP32 products of the FMA route at the edges of their tiles and forms
(plain with either transpose, symmetric A from its lower triangle, lower C).

Tolerance: the forward bound of a sum of K FP32 products in any order,
2 (K + 3) 2^-24 (|alpha| |A||B| + |beta||C0|), against FP64 products.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (127, 129, 15), (128, 64, 16), (129, 65, 17), (64, 128, 400), (63, 1000, 513), (1000, 33, 2049),
          (256, 256, 161), (257, 300, 8), (300, 259, 160), (700, 513, 333), (130, 127, 1300),
          (32, 32, 511), (64, 64, 512), (33, 100, 2051), (1, 5, 4000)]


def _mat(rows, cols, pad, g):
    return torch.randn(cols, rows + pad, dtype=torch.float32, device="cuda", generator=g)[:, :rows].t()


@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("m,n,k", SHAPES)
def test_plain(m, n, k, ta, tb):
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    A = _mat(k, m, 3, g) if ta else _mat(m, k, 1, g)
    B = _mat(n, k, 2, g) if tb else _mat(k, n, 5, g)
    a, b = (A.t() if ta else A).double(), (B.t() if tb else B).double()
    C = _mat(m, n, 1, g)
    C0 = C.double().clone()
    F.sgemm(A, B, trans_a=ta, trans_b=tb, alpha=-0.75, beta=0.5, C=C, route=0)
    ref = -0.75 * (a @ b) + 0.5 * C0
    bound = 2 * (k + 3) * 2.0 ** -24 * (0.75 * (a.abs() @ b.abs()) + 0.5 * C0.abs())
    assert torch.all((C.double() - ref).abs() <= bound)
    again = _mat(m, n, 1, g)
    again.copy_(C0)
    F.sgemm(A, B, trans_a=ta, trans_b=tb, alpha=-0.75, beta=0.5, C=again, route=0)
    assert torch.equal(again, C)  # no atomics


@pytest.mark.parametrize("m,n", [(1, 1), (127, 32), (128, 64), (129, 64), (300, 32), (1000, 64), (1025, 65), (400, 200)])
def test_symmetric_a(m, n):
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(m + n)
    A, B = _mat(m, m, 2, g), _mat(m, n, 0, g)
    low = torch.tril(A).double()
    full = low + torch.tril(low, -1).t()
    A += torch.triu(torch.full_like(A, float("nan")), 1)  # the upper triangle is not read
    C = F.sgemm(A, B, form=1, route=0)
    bound = 2 * (m + 3) * 2.0 ** -24 * (full.abs() @ B.double().abs())
    assert torch.all((C.double() - full @ B.double()).abs() <= bound)


@pytest.mark.parametrize("n,k", [(100, 30), (256, 64), (257, 128), (300, 161), (513, 200)])
def test_lower_c(n, k):
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(n + k)
    A, B = _mat(n, k, 1, g), _mat(n, k, 0, g)
    C = torch.full((n, n), 3.0, dtype=torch.float32, device="cuda").t()
    F.sgemm(A, B, trans_b=True, form=2, beta=1.0, C=C, route=0)
    ref = A.double() @ B.double().t() + 3.0
    bound = 2 * (k + 3) * 2.0 ** -24 * (A.double().abs() @ B.double().abs().t() + 3.0)
    err = (C.double() - ref).abs()
    low = torch.tril(torch.ones(n, n, dtype=torch.bool, device="cuda"))
    assert torch.all(err[low] <= bound[low]) and torch.all(C[~low] == 3.0)
