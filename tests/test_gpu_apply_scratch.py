"""Applies on a device that has room for the FP64 products' scratch but not for
the digits': served by the FP64 engine, as frac_apply is.

Tolerance: both products are sums of n terms, each term within a few eps, in any
order: 4 (n + 8) eps |V| (g (|V|^T |F|)) with g the multiplier.
"""
import contextlib

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def _room(nbytes):
    """Leaves about nbytes of the device free."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - nbytes, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del hold
        torch.cuda.empty_cache()


def _close(U, V, g, W, Wabs):
    bound = 4 * (V.shape[0] + 8) * torch.finfo(torch.float64).eps * (V.abs() @ (g * Wabs))
    assert torch.all((U - V @ (g * W)).abs() <= bound)


def test_mass_apply():
    import paper_1911_11906_gb300 as F
    n, m, k = 2000, 3, 40000
    gen = torch.Generator(device="cuda").manual_seed(1)
    V = torch.linalg.qr(torch.randn(n, n, dtype=torch.float64, device="cuda", generator=gen))[0].contiguous().t()
    theta = torch.sort(torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) + 0.5)[0]
    Fc = torch.randn(m, n, dtype=torch.float64, device="cuda", generator=gen).t()
    rowptr = torch.arange(n + 1, device="cuda")
    col, val = torch.arange(n, device="cuda").int(), torch.ones(n, dtype=torch.float64, device="cuda")
    rng = np.random.default_rng(2)
    pf, pa = rng.integers(0, m, size=k).astype(np.int32), rng.uniform(-1.0, 2.0, size=k)
    ctx = F.Context(wait_timeout_s=5.0)
    lib, p = ctx.lib, lambda t: t.data_ptr()
    need, base = lib.fraclap_apply_mass_workspace_bytes(ctx.handle, n, m, k), lib.fraclap_apply_workspace_bytes(n, m, k)
    assert need > base + (2 << 30)
    U = torch.empty(k, n, dtype=torch.float64, device="cuda").t()
    dpf, dpa = torch.from_numpy(pf).cuda(), torch.from_numpy(pa).cuda()
    with _room(base + (1 << 30)):  # no workspace given: the library's own
        ctx.check(lib.frac_apply_mass(ctx.handle, p(V), n, p(theta), n, p(rowptr), p(col), p(val), p(Fc), n, m, p(dpf), p(dpa),
                                      k, p(U), n, None, 0, None))
        ctx.sync()
        del ctx
    g = theta[:, None] ** (-dpa[None, :] / 2)
    _close(U, V, g, (V.t() @ Fc)[:, dpf.long()], (V.t().abs() @ Fc.abs())[:, dpf.long()])


def test_batched_solve():
    import paper_1911_11906_gb300 as F
    n, m, k = 800, 2, 60000
    gen = torch.Generator(device="cuda").manual_seed(3)
    Q = torch.linalg.qr(torch.randn(n, n, dtype=torch.float64, device="cuda", generator=gen))[0]
    A = (Q * torch.linspace(1.0, 2.0, n, dtype=torch.float64, device="cuda")) @ Q.t()
    A = (A + A.t()) / 2
    Fc = torch.randn(m, n, dtype=torch.float64, device="cuda", generator=gen).t()
    rng = np.random.default_rng(4)
    pf, pa = rng.integers(0, m, size=k).astype(np.int32), rng.uniform(-1.0, 2.0, size=k)
    ctx = F.Context(wait_timeout_s=5.0)
    base = ctx.lib.fraclap_apply_workspace_bytes(n, m, k)
    assert ctx.lib.fraclap_apply_workspace_bytes_ctx(ctx.handle, n, m, k) > base + (2 << 30)
    with _room(2 * base + (1 << 30)):
        (lam, V, U), = F.solve_batched([{"A": A, "F": Fc, "pair_f": pf, "pair_alpha": pa}], ctx=ctx)
        del ctx
    g = lam[:, None] ** (-torch.from_numpy(pa).cuda()[None, :] / 2)
    j = torch.from_numpy(pf).cuda().long()
    _close(U, V, g, (V.t() @ Fc)[:, j], (V.t().abs() @ Fc.abs())[:, j])
