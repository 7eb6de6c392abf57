"""Divide and conquer where its merges' orderings can go wrong: many equal and
close eigenvalues (long chains of deflating rotations), none at all, flipped
couplings, blocks at the edges of the launches.

Tolerances: backward stability, 10 n eps ||T||, with orthogonality to 10 n eps.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _check(d, e):
    import paper_1911_11906_gb300 as F
    n = len(d)
    lam, Z = F.tridiag_eig(torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda(), ctx=F.Context(wait_timeout_s=2.0))
    T = torch.from_numpy(np.diag(d) + np.diag(e, 1) + np.diag(e, -1)).cuda()
    eps, nrm = np.finfo(float).eps, float(torch.linalg.matrix_norm(T, 2))
    assert torch.all(lam[1:] >= lam[:-1])
    assert (T @ Z - Z * lam).norm() <= 10 * n * eps * max(nrm, 1e-300)
    assert (Z.t() @ Z - torch.eye(n, dtype=torch.float64, device="cuda")).norm() <= 10 * n * eps
    assert (lam - torch.linalg.eigvalsh(T)).abs().max() <= 10 * n * eps * max(nrm, 1e-300)


@pytest.mark.parametrize("n", [33, 64, 65, 129, 255, 256, 257, 513, 1000])
@pytest.mark.parametrize("kind", ["laplacian", "random", "glued", "graded", "negative", "clustered"])
def test_merges(n, kind):
    rng = np.random.default_rng(n)
    if kind == "laplacian":
        d, e = np.full(n, 2.0), np.full(n - 1, -1.0)
    elif kind == "random":
        d, e = rng.standard_normal(n), rng.standard_normal(n - 1)
    elif kind == "glued":  # copies of one block, weakly coupled: every eigenvalue nearly repeated
        d = np.tile(np.abs(np.arange(-10, 11)).astype(float), n // 21 + 1)[:n]
        e = np.where(np.arange(1, n) % 21 == 0, 1e-9, 1.0)
    elif kind == "graded":
        d, e = 10.0 ** np.linspace(0, -12, n), 0.1 * 10.0 ** np.linspace(0, -12, n)[1:]
    elif kind == "negative":
        d, e = -np.abs(rng.standard_normal(n)) * 5, -np.abs(rng.standard_normal(n - 1))
    else:
        d = np.round(rng.standard_normal(n) * 2) + 1e-14 * rng.standard_normal(n)
        e = 1e-13 * rng.standard_normal(n - 1)
    _check(d, e)
