"""Inertia counts on a cluster of CTAs per shift: the same counts, exactly, as
one CTA per shift (taken when there are more shifts than the SMs hold
clusters), for bands at the edges of the routes, ragged sizes, the pencil and a
shift with a zero pivot."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _band_matrix(n, b, seed):
    """Random symmetric CSR matrix (lower triangle stored with the upper) of half-width b."""
    rng = np.random.default_rng(seed)
    rowptr, col, val = [0], [], []
    offs = sorted({0, 1, b // 2, b - 1, b} - {-1})
    vals = {o: rng.standard_normal(n) for o in offs}
    for i in range(n):
        ent = {i: 0.25 * vals[0][i]}
        for o in offs[1:]:
            if i - o >= 0:
                ent[i - o] = vals[o][i]
            if i + o < n:
                ent[i + o] = vals[o][i + o]
        for c in sorted(ent):
            col.append(c)
            val.append(ent[c])
        rowptr.append(len(col))
    return (torch.tensor(rowptr, dtype=torch.int64).cuda(), torch.tensor(col, dtype=torch.int32).cuda(),
            torch.tensor(val, dtype=torch.float64).cuda())


@pytest.mark.parametrize("n,b", [(5, 4), (40, 16), (41, 17), (130, 16), (200, 64), (203, 65), (300, 167), (301, 168),
                                 (303, 255), (260, 259), (500, 40)])
@pytest.mark.parametrize("few", [1, 3, 15, 19, 38, 76])
def test_few_shifts_match_many(n, b, few):
    import paper_1911_11906_gb300 as F
    csr = _band_matrix(n, b, n + b)
    sig = np.random.default_rng(b).uniform(-3, 3, size=160)
    many = F.inertia_counts(*csr, sig, half_bandwidth=b).cpu()
    got = F.inertia_counts(*csr, sig[:few], half_bandwidth=b).cpu()
    assert torch.equal(got, many[:few])
    dense = torch.zeros(n, n, dtype=torch.float64)
    rp, c, v = (x.cpu() for x in csr)
    for i in range(n):
        dense[i, c[rp[i]:rp[i + 1]].long()] = v[rp[i]:rp[i + 1]]
    lam = torch.linalg.eigvalsh(dense)
    clear = [j for j in range(few) if (lam - sig[j]).abs().min() > 1e-6]  # counts of a stable factorisation
    assert sum(int(got[j]) != int((lam < sig[j]).sum()) for j in clear) <= len(clear) // 4  # no pivoting: a few may differ


def test_pencil_and_zero_pivot():
    import paper_1911_11906_gb300 as F
    from paper_1911_11906_gb300 import inputs as I
    mask = torch.from_numpy(I.square_mask(24)).cuda()
    fem = F.fem_assemble(mask, 1.0 / 25, dense=False)
    sig = np.linspace(10.0, 5000.0, 170)
    args = (fem["rowptr"], fem["col"], fem["valK"])
    many = F.inertia_counts(*args, sig, valM=fem["valM"]).cpu()
    assert torch.equal(F.inertia_counts(*args, sig[:11], valM=fem["valM"]).cpu(), many[:11])
    asm = F.fd_assemble(mask, 1.0 / 25, dense=False)
    csr = (asm["rowptr"], asm["col"], asm["val"])
    zero = float(asm["val"].max())  # the diagonal value: the first pivot is exactly zero
    assert F.inertia_counts(*csr, [zero, 100.0]).cpu().tolist()[0] == -1
    assert F.inertia_counts(*csr, [100.0] * 160 + [zero]).cpu()[0] == F.inertia_counts(*csr, [100.0, zero]).cpu()[0]
