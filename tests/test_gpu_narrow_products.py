"""FP64 products with narrow or few output tiles, against FP64 torch products.

Tolerance: the forward bound of a sum of K products in any order,
|C - C_ref| <= 2 (K + 3) eps (|alpha| |A||B| + |beta||C0|) entry by entry (both sides carry it).
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (31, 7, 33), (32, 8, 32), (33, 9, 255), (144, 3, 144), (65, 17, 4000), (700, 20, 257), (5, 800, 513),
          (2304, 5, 2303), (130, 77, 1)]


@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("m,n,k", SHAPES)
def test_narrow_products(m, n, k, ta, tb):
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(m * 7 + n * 3 + k)

    def mat(rows, cols, pad):  # column-major with a leading dimension above the row count
        return torch.randn(cols, rows + pad, dtype=torch.float64, device="cuda", generator=g)[:, :rows].t()
    A = mat(k, m, 3) if ta else mat(m, k, 3)
    B = mat(n, k, 1) if tb else mat(k, n, 1)
    a, b = (A.t() if ta else A), (B.t() if tb else B)
    eps = torch.finfo(torch.float64).eps
    got = F.dgemm(A, B, trans_a=ta, trans_b=tb)
    bound = 2 * (k + 3) * eps * (a.abs() @ b.abs())
    assert torch.all((got - a @ b).abs() <= bound)
    C = mat(m, n, 2)
    C0 = C.clone()
    F.dgemm(A, B, trans_a=ta, trans_b=tb, alpha=-1.5, beta=0.5, C=C)
    bound = 2 * (k + 3) * eps * (1.5 * (a.abs() @ b.abs()) + 0.5 * C0.abs())
    assert torch.all((C - (-1.5 * (a @ b) + 0.5 * C0)).abs() <= bound)


def test_narrow_products_are_reproducible_and_keep_non_finite_values():
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn(500, 600, dtype=torch.float64, device="cuda", generator=g).t()
    B = torch.randn(9, 500, dtype=torch.float64, device="cuda", generator=g).t()
    assert torch.equal(F.dgemm(A, B), F.dgemm(A, B))
    B[17, 2] = float("inf")
    B[3, 4] = float("nan")
    C = F.dgemm(A, B)
    assert torch.equal(torch.isnan(C), torch.isnan(A @ B)) and torch.equal(torch.isinf(C), torch.isinf(A @ B))
    assert torch.all(torch.isfinite(C[:, [0, 1, 3, 5, 6, 7, 8]]))
