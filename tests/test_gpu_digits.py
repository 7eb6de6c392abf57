"""Balanced digits of the sliced products: values at the digits' edges.

Tolerance per entry, with D digits of r bits: every operand's last digit is
rounded to 2^-rD of its row's scale 2^e <= 2 max, the dropped digit pairs
(p + q >= D) are below (D - 1) 2^-rD, so K (D + 1) 2^-rD * 4 max_a max_b; the
folds and the FP64 reference add (K + 4 D) eps |A||B|, and where a product is
subnormal up to 4 D roundings to a multiple of 2^-1074.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _digits(bits, slices, k):
    if bits == 8 or k <= 256:
        return 9, min(slices, 7)
    return 8, (slices + 1 if slices <= 5 or slices == 8 else slices)


@pytest.mark.parametrize("slices", [1, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("bits,k", [(7, 1), (7, 256), (7, 257), (7, 1024), (7, 1025), (7, 3000), (8, 257), (8, 1025)])
@pytest.mark.parametrize("ta", [True, False])
def test_digit_edges(bits, k, slices, ta):
    import paper_1911_11906_gb300 as F
    m, n = 133, 70
    g = torch.Generator(device="cuda").manual_seed(k + slices)
    # mantissas at the edges of the digits, signs and a spread of exponents inside a row
    edge = torch.tensor([1.0, 1 - 2.0 ** -53, 0.5, 0.5 + 2.0 ** -8, 255 / 256, 127.5 / 128, 1 / 3, 2.0 ** -1030, 0.0],
                        dtype=torch.float64, device="cuda")

    def draw(rows, cols):
        x = edge[torch.randint(0, edge.numel(), (cols, rows), device="cuda", generator=g)]
        x = x * torch.where(torch.rand(cols, rows, device="cuda", generator=g) < 0.5, -1.0, 1.0)
        return x * torch.exp2(torch.randint(-40, 41, (cols, rows), device="cuda", generator=g).double())
    A = draw(k, m) if ta else draw(m, k).t()  # (m, k): contiguous along k, or along m
    Bc = draw(k, n).t()  # (k, n), contiguous along k
    ctx = F.Context(wait_timeout_s=2.0)
    ctx.set_schedule("ozaki_bits", bits)
    got = F.dgemm_ozaki(A.t() if ta else A, Bc, trans_a=ta, slices=slices, ctx=ctx)
    ref = A @ Bc
    r, D = _digits(bits, slices, k)
    eps = torch.finfo(torch.float64).eps
    scale = A.abs().amax(1)[:, None] * Bc.abs().amax(0)[None, :]
    bound = 4 * k * (D + 1) * 2.0 ** (-r * D) * scale + (k + 4 * D) * eps * (A.abs() @ Bc.abs()) + 4 * D * 2.0 ** -1074
    assert torch.all((got - ref).abs() <= bound)
