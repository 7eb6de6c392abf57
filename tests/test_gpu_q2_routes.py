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
