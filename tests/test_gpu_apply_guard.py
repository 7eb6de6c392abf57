"""Default applies whose terms are small beside the largest entries of their rows
and columns: modes of separate components with forcings of different size, point
sources, strong damping.  Products formed from digits (relative to those largest
entries) must give what FP64 sums guarantee, entry by entry.

Tolerance: both products are sums of n terms, each term within a few eps, in any
order: 4 (n + 8) eps |V| (g (|V|^T |F|)) with g the multiplier.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _two_components(n, n1, g):
    V = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    for lo, hi in ((0, n1), (n1, n)):
        V[lo:hi, lo:hi] = torch.linalg.qr(torch.randn(hi - lo, hi - lo, dtype=torch.float64, device="cuda", generator=g))[0]
    return V[:, torch.randperm(n, device="cuda", generator=g)].t().contiguous().t()


def _check(F, ctx, V, lam, Fc, pf, pa, pt=None):
    n = V.shape[0]
    before = ctx.launch_count()
    if pt is None:
        U = F.frac_apply(V, lam, Fc, pf, pa, ctx=ctx)
        g = lam[:, None] ** (-torch.from_numpy(pa).cuda()[None, :] / 2)
    else:
        U = F.frac_diffusion(V, lam, Fc, pf, pa, pt, ctx=ctx)
        g = torch.exp(-lam[:, None] ** (torch.from_numpy(pa).cuda()[None, :] / 2) * torch.from_numpy(pt).cuda()[None, :])
    assert ctx.launch_count() - before > 3  # the digits' route
    j = torch.from_numpy(pf).cuda().long()
    ref = V @ (g * (V.t() @ Fc)[:, j])
    bound = 4 * (n + 8) * torch.finfo(torch.float64).eps * (V.abs() @ (g * (V.t().abs() @ Fc.abs())[:, j]))
    assert torch.all((U - ref).abs() <= bound)


@pytest.mark.parametrize("scale", [1.0, 1e10, 1e17, 1e20, 1e200])
@pytest.mark.parametrize("n,n1,m,k", [(1025, 400, 300, 701), (250, 113, 3000, 2900), (2049, 2048, 65, 129)])
def test_separate_components(n, n1, m, k, scale):
    import paper_1911_11906_gb300 as F
    g = torch.Generator(device="cuda").manual_seed(n)
    V = _two_components(n, n1, g)
    lam = torch.sort(torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * 1e5 + 20.0)[0]
    Fc = torch.randn(m, n, dtype=torch.float64, device="cuda", generator=g)
    Fc[::2, :n1] *= scale
    rng = np.random.default_rng(n)
    _check(F, F.Context(wait_timeout_s=2.0), V, lam, Fc.t(), rng.integers(0, m, size=k).astype(np.int32), rng.uniform(-1.0, 2.0, size=k))


def test_point_sources_zero_columns_and_damping():
    import paper_1911_11906_gb300 as F
    n, m, k = 1025, 300, 701
    g = torch.Generator(device="cuda").manual_seed(11)
    i = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
    V = (torch.sin(torch.pi / (n + 1) * torch.outer(i, i) % (2 * torch.pi)) * (2.0 / (n + 1)) ** 0.5).t()
    lam = 4.0 * (n + 1) ** 2 * torch.sin(torch.pi / 2 / (n + 1) * i) ** 2
    Fc = torch.zeros(m, n, dtype=torch.float64, device="cuda")
    Fc[torch.arange(m), torch.randint(0, n, (m,), device="cuda", generator=g)] = 1.0  # one node each
    Fc[1::4] += 1e-25 * torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    Fc[2::4] = 0.0
    rng = np.random.default_rng(12)
    pf, pa = rng.integers(0, m, size=k).astype(np.int32), rng.uniform(0.1, 1.9, size=k)
    ctx = F.Context(wait_timeout_s=2.0)
    _check(F, ctx, V, lam, Fc.t(), pf, pa)
    _check(F, ctx, V, lam, Fc.t(), pf, pa, rng.uniform(1e-4, 0.4, size=k))
