"""FP64 products with more columns than one launch of the narrow kernels takes.

Tolerance: the forward bound of a sum of K products in any order, as in the
narrow products' test.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

LAUNCH = 65535 * 8  # columns of one launch


@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (False, True)])
@pytest.mark.parametrize("m,n,k", [(32, 600000, 17), (3, 2 * LAUNCH + 1, 1), (33, LAUNCH, 9), (33, LAUNCH + 1, 9)])
def test_products_of_many_columns(m, n, k, ta, tb):
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(m + k)
    mat = lambda rows, cols: torch.randn(cols, rows, dtype=torch.float64, device="cuda", generator=g).t()  # noqa: E731
    A, B, C = (mat(k, m) if ta else mat(m, k)), (mat(n, k) if tb else mat(k, n)), mat(m, n)
    a, b, C0 = (A.t() if ta else A), (B.t() if tb else B), C.clone()
    F.dgemm(A, B, trans_a=ta, trans_b=tb, alpha=-1.5, beta=0.5, C=C)
    bound = 2 * (k + 3) * torch.finfo(torch.float64).eps * (1.5 * (a.abs() @ b.abs()) + 0.5 * C0.abs())
    assert torch.all((C - (-1.5 * (a @ b) + 0.5 * C0)).abs() <= bound)


def test_apply_of_many_forcings():
    import paper_1911_11906_gb300 as F
    n, m, k = 12, 600000, 40
    g = torch.Generator(device="cuda").manual_seed(3)
    V = torch.linalg.qr(torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g))[0].t()
    lam = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
    Fc = torch.randn(m, n, dtype=torch.float64, device="cuda", generator=g).t()
    pf = (m - 1 - 14999 * torch.arange(k, device="cuda")).int()
    U = F.frac_apply(V, lam, Fc, pf, torch.full((k,), 2.0, dtype=torch.float64, device="cuda"), ctx=F.Context(wait_timeout_s=2.0))
    ref = V @ ((V.t() @ Fc[:, pf.long()]) / lam[:, None])
    bound = 4 * (n + 8) * torch.finfo(torch.float64).eps * (V.abs() @ ((V.t().abs() @ Fc[:, pf.long()].abs()) / lam[:, None]))
    assert torch.all((U - ref).abs() <= bound)
