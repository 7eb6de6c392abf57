"""Blocked stage-2 back-transformation at the edges of its blocks (b reflectors
of consecutive sweeps, windows of 2b rows, 8 to 64 columns per CTA).

Tolerances: a product of O(n) Householder reflectors is orthogonal, and the
similarity it forms backward stable, to a modest multiple of n eps; 10 n eps
(relative to ||A||_F for the similarity) is used.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b", [32, 64])
@pytest.mark.parametrize("n", [2, 3, 33, 34, 64, 65, 66, 97, 128, 129, 130, 193, 300, 517])
def test_q_reconstructs_a(n, b):
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(n + b)
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    A = A + A.t()
    eps = torch.finfo(torch.float64).eps
    d, e, Q = F.tridiagonalize(A, ctx=F.Context(band_width=b, wait_timeout_s=2.0))
    T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
    assert (Q.t() @ Q - torch.eye(n, dtype=torch.float64, device="cuda")).norm() <= 10 * n * eps
    assert (Q @ T @ Q.t() - A).norm() <= 10 * n * eps * A.norm()


@pytest.mark.parametrize("n", [150, 700])
def test_blocks_agree_with_single_reflectors(n):
    """The reflector-by-reflector kernel (the q2_parts knob) gives the same Q to rounding."""
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    A = A + A.t()
    eps = torch.finfo(torch.float64).eps
    blocks, single = F.Context(band_width=64), F.Context(band_width=64)
    single.set_schedule("q2_parts", 8)
    # the same band and reflectors up to rounding; Q's columns are compared through what they diagonalise
    for ctx in (blocks, single):
        d, e, Q = F.tridiagonalize(A, ctx=ctx)
        T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
        assert (Q @ T - A @ Q).norm() <= 10 * n * eps * A.norm()


@pytest.mark.parametrize("b,m", [(32, 20), (32, 33), (64, 20), (64, 47)])
def test_mixed_route_on_blocks(b, m):
    """FP32 blocks: the refined decomposition meets the FP64 bars (residual and orthogonality)."""
    import numpy as np
    import paper_1911_11906_gb300 as F
    from paper_1911_11906_gb300 import inputs as I
    ctx = F.Context(band_width=b, wait_timeout_s=2.0)
    mask = I.ellipse_mask(m, 6, np.random.default_rng(m))
    asm = F.fd_assemble(torch.from_numpy(mask).cuda(), 1.0 / (m + 1), ctx=ctx)
    lam, V = F.eig_full_mixed(asm["A"], asm["rowptr"], asm["col"], asm["val"], refine_iters=6, ctx=ctx)
    A, n = asm["A"], asm["n"]
    assert (A @ V - V * lam).norm() / (A.norm() * n) <= 1e-13
    assert (V.t() @ V - torch.eye(n, dtype=torch.float64, device="cuda")).abs().max() <= 1e-12
    # the FP32 stages start the refinement no further off than single reflectors would: O(n eps32)
    assert ctx.refine_stats()[0]["norm2_R"] <= 10 * n * 2.0 ** -24
