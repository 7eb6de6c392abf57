"""Panels of the band reduction at the edges of their splits: CTAs of a cluster
(48 or 128 rows at least, 16 at most), rows a thread keeps, panels lower than
they are wide, columns that are zero below the diagonal.

Tolerances: a product of O(n) Householder reflectors is orthogonal, and the
similarity it forms backward stable, to a modest multiple of n eps; 10 n eps
(relative to ||A||_F for the similarity) is used, eps = 2^-52 (FP64 stages) or
2^-23 (FP32 stages, read from the first refinement step's residuals).
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _check64(A, b):
    import paper_1911_11906_gb300 as F
    n, eps = A.shape[0], torch.finfo(torch.float64).eps
    d, e, Q = F.tridiagonalize(A, ctx=F.Context(band_width=b, wait_timeout_s=2.0))
    T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
    assert (Q.t() @ Q - torch.eye(n, dtype=torch.float64, device="cuda")).norm() <= 10 * n * eps
    assert (Q @ T @ Q.t() - A).norm() <= 10 * n * eps * A.norm()


@pytest.mark.parametrize("n,b", [(9, 8), (48, 32), (81, 32), (112, 64), (113, 64), (161, 32), (1025 + 32, 32),
                                 (1537 + 64, 64), (2049 + 32, 32)])
def test_fp64_panels(n, b):
    g = torch.Generator(device="cuda").manual_seed(n + b)
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    _check64(A + A.t(), b)


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -300, 2.0 ** 300])
def test_fp64_zero_columns(scale):
    g = torch.Generator(device="cuda").manual_seed(7)
    A = torch.randn(200, 200, dtype=torch.float64, device="cuda", generator=g) * scale
    A = A + A.t()
    A[10:50] = 0  # rows and columns without any entry but the diagonal's
    A[:, 10:50] = 0
    A.diagonal()[10:50] = scale
    _check64(A, 32)


@pytest.mark.parametrize("n,b", [(40, 32), (70, 64), (128 + 32, 32), (129 + 64, 64), (2049 + 64, 64), (2049 + 32, 32),
                                 (4097 + 64, 64), (6145 + 64, 64), (8193 + 64, 64)])
def test_fp32_panels(n, b):
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(n + b)
    # a few random symmetric entries a row on a spread diagonal
    i = torch.arange(n, device="cuda").repeat(3)
    j = torch.randint(0, n, (3 * n,), device="cuda", generator=g)
    v = torch.randn(3 * n, dtype=torch.float64, device="cuda", generator=g)
    A = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    A.index_put_((i, j), v, accumulate=True)
    A = A + A.t() + torch.diag(torch.linspace(1.0, 20.0, n, dtype=torch.float64, device="cuda"))
    rows, cols = torch.nonzero(A, as_tuple=True)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    ctx = F.Context(band_width=b, wait_timeout_s=2.0)
    lam, V = F.eig_full_mixed(A, rowptr, cols.to(torch.int32), A[rows, cols].contiguous(), refine_iters=6, ctx=ctx)
    first = ctx.refine_stats()[0]
    assert first["fro_R"] <= 10 * n * 2.0 ** -23
    assert (A @ V - V * lam).norm() <= 1e-13 * n * A.norm()
    assert (V.t() @ V - torch.eye(n, dtype=torch.float64, device="cuda")).abs().max() <= 1e-12
