"""The pencil's banded solves at the edges of their windows (32 positions of a
lane's register, half-bandwidths up to 256 in registers, a ring past that).

Tolerance: M's diagonal lies in [1, 1.25] and its off-diagonal row sums below
1/2, so its condition number is below 4 and every step is backward stable to a
modest multiple of n eps; 50 n eps relative to the norms is used.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,b", [(1, 0), (2, 1), (31, 30), (32, 0), (33, 32), (64, 31), (65, 33), (97, 64), (130, 65),
                                 (300, 255), (300, 256), (300, 257), (301, 300), (515, 96), (515, 129)])
def test_pencil_of_band(n, b):
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(1000 * n + b)
    i = torch.arange(n, device="cuda")
    d = (i[:, None] - i[None, :]).abs()
    M = torch.rand(n, n, dtype=torch.float64, device="cuda", generator=g) * (d <= b) * (d > 0) / (4 * max(b, 1))
    M = (M + M.t()) / 2  # off-diagonal entries below 1 / (4 b), row sums below 1 / 2
    M = M + torch.eye(n, dtype=torch.float64, device="cuda") * (1 + torch.rand(n, dtype=torch.float64, device="cuda", generator=g) / 4)
    K = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    K = K + K.t()
    rows, cols = torch.nonzero(d <= b, as_tuple=True)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    theta, Phi = F.eig_pencil(K, rowptr, cols.to(torch.int32), M[rows, cols].contiguous(), half_bandwidth=b,
                              ctx=F.Context(wait_timeout_s=2.0))
    eps = torch.finfo(torch.float64).eps
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    assert (Phi.t() @ M @ Phi - eye).norm() <= 50 * n * eps
    assert (K @ Phi - (M @ Phi) * theta).norm() <= 50 * n * eps * K.norm()
