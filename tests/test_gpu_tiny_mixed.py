"""The mixed route on the smallest problems, whose refinement keeps more scratch
than n x n, on workspaces of exactly the size asked for with a guard behind.

Tolerances: eigenvalues to 100 eps of the largest, orthogonality to 100 eps.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("band", [8, 64])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 7, 16])
def test_tiny_mixed(n, band):
    import paper_1911_11906_gb300 as F
    ctx = F.Context(band_width=band, wait_timeout_s=2.0)
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    A = A + A.t() + 10 * n * torch.eye(n, dtype=torch.float64, device="cuda")
    rowptr = torch.arange(0, n * n + 1, n, device="cuda")
    col, val = torch.arange(n, device="cuda").int().repeat(n), A.reshape(-1).contiguous()
    need = (ctx.lib.fraclap_eig_mixed_workspace_bytes(ctx.handle, n) + 255) // 256 * 256
    ws = torch.full((need + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
    lam, V = torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty(n, n, dtype=torch.float64, device="cuda")
    p = lambda t: t.data_ptr()  # noqa: E731
    ctx.check(ctx.lib.eig_full_mixed(ctx.handle, p(A), n, n, p(rowptr), p(col), p(val), 6, p(lam), p(V), n, p(ws), need, None, None))
    ctx.sync()
    eps = torch.finfo(torch.float64).eps
    ref = torch.linalg.eigvalsh(A)
    assert torch.all((lam - ref).abs() <= 100 * eps * ref.abs().max())
    assert torch.all((V @ V.t() - torch.eye(n, dtype=torch.float64, device="cuda")).abs() <= 100 * eps)
    assert torch.all(ws[need:] == 0x5A)
