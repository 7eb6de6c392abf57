"""Workspace sizes of the eigensolvers, and back-transformations in several pieces.

The sizes count what the stages hold at one time, in entries of the working type:
the matrix, the panels (n^2 / 2), the reflectors, the divide and conquer's four
square buffers; everything else is O(n b) or n^2 / b.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("band", [8, 32, 64])
@pytest.mark.parametrize("n", [1, 40, 2304, 31996, 64081])
def test_workspace_of_the_eigensolvers(n, band):
    import paper_1911_11906_gb300 as F
    ctx = F.Context(band_width=band, wait_timeout_s=2.0)
    small = 16 * n * band + 3 * n * (n + band) // band + 8 * band * band
    two_stage = 6.5 * n * n + 8 * n + small  # working type
    if n * n // 2 * 4 <= 64 << 20:  # V T kept beside V
        two_stage += n * n / 2
    assert ctx.lib.fraclap_eig_workspace_bytes(ctx.handle, n) <= 8 * two_stage + 400 * n + 200000
    # mixed: the same in FP32 with its vectors (1) and split operands (6), and the
    # refinement: 8.5 FP64 squares, 64 x 64 blocks for n / 2 clusters and the FP64
    # eigensolver of a cluster
    refine = 8.5 * n * n + 1.5 * 64 * 64 * (n + 2) + two_stage
    assert ctx.lib.fraclap_eig_mixed_workspace_bytes(ctx.handle, n) <= 4 * (two_stage + 7 * n * n + 1600 * n) + 8 * refine + 800 * n + 3000000


@pytest.mark.parametrize("band", [32, 64])
@pytest.mark.parametrize("n", [2, 33, 64, 65, 130, 700, 1111])
def test_block_factors_a_few_steps_at_a_time(n, band):
    """The library's own workspace of tridiagonalize holds one step of the block
    factors, the eigensolver's all of them: the same Q."""
    import paper_1911_11906_gb300 as F
    ctx = F.Context(band_width=band, wait_timeout_s=2.0)
    g = torch.Generator(device="cuda").manual_seed(n + band)
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    A = A + A.t()
    d, e, Q = F.tridiagonalize(A, ctx=ctx)  # with the eigensolver's workspace
    whole = ctx.launch_count()
    d2, e2, Q2 = (torch.empty(c, dtype=torch.float64, device="cuda") for c in (n, n, n * n))
    own = F.Context(band_width=band, wait_timeout_s=2.0)
    p = lambda t: t.data_ptr()  # noqa: E731
    own.check(own.lib.fraclap_tridiagonalize(own.handle, p(A), n, n, p(d2), p(e2), p(Q2), n, None, 0, None))
    own.sync()
    steps = (n - 2) // band + 1
    assert own.launch_count() > whole or steps <= 3  # in more pieces
    assert torch.equal(Q2.view(n, n).t(), Q) and torch.equal(d2, d) and torch.equal(e2[:n - 1], e[:n - 1])
    T = torch.diag(d) + torch.diag(e[:n - 1], 1) + torch.diag(e[:n - 1], -1)
    eps = torch.finfo(torch.float64).eps
    assert torch.linalg.matrix_norm(Q.t() @ Q - torch.eye(n, dtype=torch.float64, device="cuda")) <= 20 * n * eps
    assert torch.linalg.matrix_norm(Q @ T @ Q.t() - A) <= 20 * n * eps * torch.linalg.matrix_norm(A)
