"""FP64 applies (apply_slices = 0) that are formed from digits, beside the FP64
engine (taken with the smaller documented workspace).

Tolerance, entry by entry: both products are sums of n terms, each term within
a few eps, in any order: 4 (n + 8) eps |V| (g (|V|^T |F|)) with g the multiplier.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _inputs(n, m, k, seed, wide=False):
    g = torch.Generator(device="cuda").manual_seed(seed)
    V = torch.linalg.qr(torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g))[0].t()  # column-major
    lam = torch.sort(torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * 1e5 + 20.0)[0]
    Fc = torch.randn(m, n, dtype=torch.float64, device="cuda", generator=g)
    if wide:  # entries of one column over 24 decades
        Fc = Fc * 10.0 ** (24 * torch.rand(m, n, dtype=torch.float64, device="cuda", generator=g) - 12)
    rng = np.random.default_rng(seed)
    return V, lam, Fc.t(), rng.integers(0, m, size=k).astype(np.int32), rng.uniform(-1.0, 2.0, size=k)


def _engine(F, ctx, V, lam, Fc, pf, pa):
    n, m, k = V.shape[0], Fc.shape[1], len(pf)
    ws = torch.empty(ctx.lib.fraclap_apply_workspace_bytes(n, m, k), dtype=torch.uint8, device="cuda")
    return F.frac_apply(V, lam, Fc, pf, pa, ctx=ctx, workspace=ws)


@pytest.mark.parametrize("n,m,k,wide", [(250, 3000, 2900, False), (1025, 300, 700, False), (1500, 1, 400, False),
                                        (2049, 65, 129, False), (2049, 65, 129, True)])
def test_digits_are_fp64_accurate(n, m, k, wide):
    import paper_1911_11906_gb300 as F
    ctx = F.Context(wait_timeout_s=2.0)
    V, lam, Fc, pf, pa = _inputs(n, m, k, n + k, wide)
    assert ctx.lib.fraclap_apply_workspace_bytes_ctx(ctx.handle, n, m, k) > \
        ctx.lib.fraclap_apply_workspace_bytes(n, m, k)  # the digits' route
    before = ctx.launch_count()
    U = F.frac_apply(V, lam, Fc, pf, pa, ctx=ctx)
    assert ctx.launch_count() - before > 3
    before = ctx.launch_count()
    E = _engine(F, ctx, V, lam, Fc, pf, pa)
    assert ctx.launch_count() - before == 3  # two products and the scaling
    g = lam[:, None] ** (-torch.from_numpy(pa).cuda()[None, :] / 2)
    j = torch.from_numpy(pf).cuda().long()
    ref = V @ (g * (V.t() @ Fc)[:, j])
    bound = 4 * (n + 8) * torch.finfo(torch.float64).eps * (V.abs() @ (g * (V.t().abs() @ Fc.abs())[:, j]))
    assert torch.all((U - ref).abs() <= bound) and torch.all((E - ref).abs() <= bound)


def test_non_finite_inputs_take_the_engine():
    """A column with an infinity or NaN gives what the FP64 engine gives, bit for bit."""
    import paper_1911_11906_gb300 as F
    ctx = F.Context(wait_timeout_s=2.0)
    V, lam, Fc, pf, pa = _inputs(1025, 70, 300, 5)
    for bad in (float("inf"), float("nan")):
        X = Fc.t().clone().t()
        X[17, 3] = bad
        U, E = F.frac_apply(V, lam, X, pf, pa, ctx=ctx), _engine(F, ctx, V, lam, X, pf, pa)
        assert torch.equal(torch.nan_to_num(U, nan=7.0), torch.nan_to_num(E, nan=7.0))
        assert torch.equal(torch.isnan(U), torch.isnan(E)) and not torch.all(torch.isfinite(U))


def test_graph_and_diffusion_by_digits():
    import paper_1911_11906_gb300 as F
    ctx = F.Context(wait_timeout_s=2.0)
    V, lam, Fc, pf, pa = _inputs(1025, 70, 300, 6)
    pa = np.abs(pa)
    pt = np.random.default_rng(1).uniform(0.0, 1e-3, size=300)
    U = F.frac_diffusion(V, lam, Fc, pf, pa, pt, ctx=ctx)
    G = F.ApplyGraph(V, lam, Fc, pf, pa, pair_t=pt, ctx=ctx)
    assert G.kernels > 3 and torch.equal(G.launch(), U)
    G.F[5, 5] = float("nan")
    assert torch.isnan(G.launch()).any()
    G.F[5, 5] = 1.0
    assert torch.all(torch.isfinite(G.launch()))
