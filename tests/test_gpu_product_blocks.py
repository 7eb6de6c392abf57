"""Sliced products whose digit planes do not fit beside the digits: C is formed
in blocks.  The integer sums are exact, so an entry has the same bits whatever
the block, and pieces that fit in one block are compared bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k,route", [(13000, 13001, 70, 1), (700001, 300, 70, 1), (700001, 300, 70, 0)])
def test_blocks_have_the_bits_of_pieces(m, n, k, route):
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(m)
    A = torch.randn(m, k, dtype=torch.float64, device="cuda", generator=g)  # row-major: op(A) = A.t() transposed
    Bc = torch.randn(n, k, dtype=torch.float64, device="cuda", generator=g).t()
    C = torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()
    ctx = F.Context(wait_timeout_s=5.0)
    ctx.set_tensor_route(route)
    got = F.dgemm_ozaki(A.t(), Bc, trans_a=True, alpha=-1.5, beta=0.25, C=C.t().clone().t(), ctx=ctx)
    for i0, i1 in ((0, 1500), (m // 2 - 700, m // 2 + 900), (m - 1100, m)):
        for j0, j1 in ((0, 200), (n // 2 - 140, n // 2 + 150), (n - 130, n)):
            piece = F.dgemm_ozaki(A[i0:i1].t(), Bc[:, j0:j1].t().contiguous().t(), trans_a=True, alpha=-1.5, beta=0.25,
                                  C=C[i0:i1, j0:j1].t().contiguous().t(), ctx=ctx)
            assert torch.equal(got[i0:i1, j0:j1], piece)
    ref = -1.5 * (A @ Bc) + 0.25 * C
    bound = 4 * (k + 28) * torch.finfo(torch.float64).eps * (1.5 * (A.abs() @ Bc.abs()) + C.abs())
    assert torch.all((got - ref).abs() <= bound)
