"""The two routes of the stage-2 back-transformation on the same reduction: blocks of
reflectors and the reflectors one by one give the same Q, and each Q is orthogonal.

Tolerance: either route multiplies O(n) orthogonal factors, so both are within 10 n
eps (Frobenius norm) of the exact product, and within 20 n eps of each other.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 65, 66, 150, 700, 1300])
def test_blocks_and_single_reflectors_give_the_same_q(n):
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    A = A + A.t()
    eps, eye = torch.finfo(torch.float64).eps, torch.eye(n, dtype=torch.float64, device="cuda")
    out = []
    for parts in (0, 8, 16):
        ctx = F.Context(band_width=64, wait_timeout_s=2.0)
        ctx.set_schedule("q2_parts", parts)
        out.append(F.tridiagonalize(A, ctx=ctx))
        assert (out[-1][2].t() @ out[-1][2] - eye).norm() <= 10 * n * eps
    for d, e, Q in out[1:]:
        assert torch.equal(d, out[0][0]) and torch.equal(e, out[0][1])  # the reduction is shared
        assert (Q - out[0][2]).norm() <= 20 * n * eps


@pytest.mark.parametrize("band", [32, 64])
def test_fp64_routes_of_many_columns(band):
    """Past 4096 columns the first back-transformation splits its sums, past 4256 the
    second applies reflectors one by one (b = 64): residual and orthogonality of the
    whole FP64 decomposition, to 10 n eps."""
    import paper_1911_11906_gb300 as F
    n, eps = 4300, torch.finfo(torch.float64).eps
    g = torch.Generator(device="cuda").manual_seed(band)
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    A = A + A.t()
    lam, V = F.eig_full(A, ctx=F.Context(band_width=band, wait_timeout_s=5.0))[:2]
    assert (V.t() @ V - torch.eye(n, dtype=torch.float64, device="cuda")).norm() <= 10 * n * eps
    assert (A @ V - V * lam).norm() <= 10 * n * eps * A.norm()
