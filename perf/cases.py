"""The work this library is used for, as a list of cases with sizes.

Kinds of case (field "kind"):

* "apply": the spectral solution operator on a decomposition that a program
  keeps (`frac_apply`, `frac_diffusion` when "times" is set, or the captured
  `ApplyGraph` when "graph" is set).  V and lambda are the closed-form sine
  modes of an nx x ny rectangle, the eigenvectors of the same 5-point operator
  that the decomposition entry points diagonalise, so a state costs no solve.
* "solve": the whole path on a masked grid: `fd_assemble`, all eigenpairs
  (`eig_full`, or `eig_full_mixed` with the CSR form), `frac_apply`.
* "batch": many uneven small problems through `solve_batched`.
* "fem": `fem_assemble`, `eig_pencil`, `frac_apply_mass`.
* "product": `dgemm_ozaki`, the FP64-accurate product behind the refinement.
* "counts": `inertia_counts` at many shifts (spectrum slicing).

A decomposition's eigenvectors are not returned by themselves: the sign of
each, and the basis inside a multiple eigenvalue, are unspecified.  Every one
of them enters the solutions U, which are returned whole, as are the
eigenvalues.  Masks, forcings and orders are drawn from the seed; a mask is
cut to exactly the case's number of unknowns, so a case is the same amount of
work whatever the seed.
"""
import math

import numpy as np
import torch

import paper_1911_11906_gb300 as F
from paper_1911_11906_gb300 import inputs as I

_contexts = {}


def _context(band_width=0, slices=0):
    """A program makes one context per configuration and keeps it."""
    key = (band_width, slices)
    if key not in _contexts:
        ctx = F.Context(band_width=band_width)
        ctx.set_apply_slices(slices)
        _contexts[key] = ctx
    return _contexts[key]


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def listed():
    return [
        # the smoke-sized apply: a handful of solves on a tiny grid, all launch latency
        {"name": "apply_144", "kind": "apply", "nx": 12, "ny": 12, "m": 3, "k": 9, "slices": 0, "times": False, "graph": False},
        # the 48 x 48 square's 5 forcings x 4 orders replayed as one captured graph (a time loop)
        {"name": "graph_2304", "kind": "apply", "nx": 48, "ny": 48, "m": 5, "k": 20, "slices": 0, "times": False, "graph": True},
        # 16 forcings x 8 orders at the size of the 128 x 128 ellipse grid, the default FP64 products, odd extents
        {"name": "apply_8835_fp64", "kind": "apply", "nx": 95, "ny": 93, "m": 16, "k": 128, "slices": 0, "times": False, "graph": False},
        # fractional diffusion: 7 initial states x 11 orders at one time each, sliced products at FP64 level, odd n
        {"name": "diffusion_2867_s7", "kind": "apply", "nx": 61, "ny": 47, "m": 7, "k": 77, "slices": 7, "times": True, "graph": False},
        # the apply at scale: one order per distinct forcing, 4096 of them, sliced products
        {"name": "apply_18225_s6", "kind": "apply", "nx": 135, "ny": 135, "m": 4096, "k": 4096, "slices": 6, "times": False, "graph": False},
        # the flagship: 128 x 128 six-ellipse grid, 16 forcings x 8 orders, mixed route
        {"name": "solve_8810_mixed", "kind": "solve", "route": "mixed", "dim": 2, "grid": 128, "n": 8810, "m": 16, "orders": 8},
        # a small holed cube (7-point, clustered spectrum), mixed route, odd n
        {"name": "solve_3001_cube_mixed", "kind": "solve", "route": "mixed", "dim": 3, "grid": 15, "n": 3001, "m": 8, "orders": 4},
        # the 48 x 48 square, 5 forcings x 4 orders, FP64 throughout
        {"name": "solve_2304_fp64", "kind": "solve", "route": "fp64", "dim": 2, "grid": 48, "n": 2304, "m": 5, "orders": 4},
        # many uneven small problems (sides 20 to 64), 8 forcings x 4 orders each
        {"name": "batch_32", "kind": "batch", "count": 32, "side_lo": 20, "side_hi": 64, "m": 8, "orders": 4},
        # the generalised problem with a mass matrix on a small domain
        {"name": "fem_751", "kind": "fem", "grid": 40, "n": 751, "m": 8, "orders": 4},
        # the refinement's residual product X^T Y, full accuracy, ragged in every extent
        {"name": "product_4099", "kind": "product", "rows": 4099, "cols": 4031, "inner": 4157, "slices": 7},
        # slicing the flagship's spectrum: exact counts at 15 shifts
        {"name": "counts_8810", "kind": "counts", "grid": 128, "n": 8810, "shifts": 15},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply"] * 5 + ["solve"] * 5 + ["batch", "fem", "product", "product", "counts"])
    if kind == "apply":
        while True:
            nx, ny = _log_int(rng, 11, 135), _log_int(rng, 11, 135)
            slices = rng.choice([0, 0, 6, 7])
            m, k = _log_int(rng, 1, 4096), _log_int(rng, 1, 4096)
            if 2.0 * (nx * ny) ** 2 * (m + k) <= (2e11 if slices == 0 else 5e12):
                break
        return {"kind": kind, "nx": nx, "ny": ny, "m": m, "k": k, "slices": slices, "times": rng.random() < 0.4,
                "graph": rng.random() < 0.2}
    if kind == "solve":
        if rng.random() < 0.3:
            n = _log_int(rng, 150, 2500)
            return {"kind": kind, "route": "fp64", "dim": 2, "grid": math.isqrt(2 * n) + 1, "n": n, "m": _log_int(rng, 1, 16),
                    "orders": rng.randint(1, 8)}
        n = _log_int(rng, 300, 8000)
        if n <= 4500 and rng.random() < 0.35:
            grid = 8
            while 0.85 * grid ** 3 < n:
                grid += 1
            return {"kind": kind, "route": "mixed", "dim": 3, "grid": grid, "n": n, "m": _log_int(rng, 1, 32), "orders": rng.randint(1, 8)}
        return {"kind": kind, "route": "mixed", "dim": 2, "grid": math.isqrt(2 * n) + 1, "n": n, "m": _log_int(rng, 1, 32),
                "orders": rng.randint(1, 8)}
    if kind == "batch":
        lo = rng.randint(18, 30)
        return {"kind": kind, "count": _log_int(rng, 3, 40), "side_lo": lo, "side_hi": rng.randint(lo + 5, 64), "m": _log_int(rng, 1, 16),
                "orders": rng.randint(1, 4)}
    if kind == "fem":
        n = _log_int(rng, 100, 900)
        return {"kind": kind, "grid": math.isqrt(2 * n) + 1, "n": n, "m": _log_int(rng, 1, 16), "orders": rng.randint(1, 4)}
    if kind == "product":
        return {"kind": kind, "rows": _log_int(rng, 130, 6000), "cols": _log_int(rng, 20, 6000), "inner": _log_int(rng, 130, 6000),
                "slices": rng.choice([5, 6, 7])}
    n = _log_int(rng, 400, 8000)
    return {"kind": kind, "grid": math.isqrt(2 * n) + 1, "n": n, "shifts": _log_int(rng, 1, 40)}


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _mask(dim, grid, n, seed):
    """A random domain of exactly n nodes: drawn until it has at least n, then
    cut at its n-th node in dof order.  grid, n = 48, 2304 is the full square."""
    if dim == 2 and n == grid * grid:
        return I.square_mask(grid)
    for attempt in range(1000):
        rng = np.random.default_rng([seed, attempt])
        mask = I.ellipse_mask(grid, 6, rng) if dim == 2 else I.holed_cube_mask(grid, 5, rng)
        if int(mask.sum()) >= n:
            break
    else:
        raise ValueError(f"no domain of {n} nodes on this grid")
    flat = mask.reshape(-1)
    flat[np.flatnonzero(flat)[n:]] = 0
    return mask


def _forcings(mask, m, seed):
    """Cubic polynomials and, every other one, noise at the nodes; column-major on the GPU."""
    h = 1.0 / (mask.shape[0] + 1)
    coords = I.dof_coords(mask, h)
    rng = np.random.default_rng([seed, 7])
    cols = [I.poly_forcing(coords, rng) if j % 2 == 0 else rng.standard_normal(coords.shape[0]) for j in range(m)]
    return torch.from_numpy(np.ascontiguousarray(np.stack(cols))).cuda().t()


def _pairs(m, orders, seed):
    alphas = np.random.default_rng([seed, 9]).uniform(0.1, 2.0, size=orders)
    pf, pa = np.repeat(np.arange(m, dtype=np.int32), orders), np.tile(alphas, m)
    return torch.from_numpy(pf).cuda(), torch.from_numpy(pa).cuda()


def _sides(case):
    c = case["count"]
    return [case["side_lo"] + (case["side_hi"] - case["side_lo"]) * i // max(c - 1, 1) for i in range(c)]


def _rectangle(nx, ny):
    """(lambda ascending, V column-major): the sine modes of the nx x ny grid of spacing 1 / (max + 1)."""
    def modes(c):
        i = torch.arange(1, c + 1, dtype=torch.float64, device="cuda")
        return torch.sin(math.pi / (c + 1) * torch.outer(i, i) % (2 * math.pi)) * math.sqrt(2.0 / (c + 1)), torch.sin(math.pi / 2 / (c + 1) * i) ** 2
    (sx, lx), (sy, ly) = modes(nx), modes(ny)
    lam, order = (4.0 * (max(nx, ny) + 1) ** 2 * (ly[:, None] + lx[None, :])).reshape(-1).sort()
    rows = torch.einsum("jy,ix->jiyx", sy, sx).reshape(nx * ny, nx * ny)[order]  # one mode per row
    return lam, rows.contiguous().t()


def _apply_inputs(case, seed):
    n, m, k = case["nx"] * case["ny"], case["m"], case["k"]
    lam, V = _rectangle(case["nx"], case["ny"])
    g = torch.Generator(device="cuda").manual_seed(seed)
    cols = torch.randn(m, n, dtype=torch.float64, device="cuda", generator=g)
    y = (torch.arange(n, device="cuda") // case["nx"] + 1.0).double() / (case["ny"] + 1)
    x = (torch.arange(n, device="cuda") % case["nx"] + 1.0).double() / (case["nx"] + 1)
    powers = torch.stack([x ** a * y ** b for a in range(4) for b in range(4 - a)])
    half = (m + 1) // 2
    cols[::2] = torch.randn(half, 10, dtype=torch.float64, device="cuda", generator=g) @ powers  # every other forcing a cubic
    r = np.random.default_rng([seed, 11])
    pf = np.arange(k) % m if k >= m else r.integers(0, m, size=k)
    pa, pt = r.uniform(0.1, 1.9, size=k), r.uniform(1e-4, 0.4, size=k)
    return lam, V, cols.t(), torch.from_numpy(pf.astype(np.int32)).cuda(), torch.from_numpy(pa).cuda(), torch.from_numpy(pt).cuda()


def _product_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    make = lambda c: torch.randn(c, case["inner"], dtype=torch.float64, device="cuda", generator=g).t() / math.sqrt(case["inner"])  # noqa: E731
    return make(case["rows"]), make(case["cols"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "apply":
        lam, V, f, pf, pa, pt = _apply_inputs(case, seed)
        ctx = _context(0, case["slices"])
        state = {"kind": kind, "ctx": ctx, "lam": lam, "V": V, "F": f, "pf": pf, "pa": pa, "pt": pt if case["times"] else None, "graph": None}
        if case["graph"]:
            state["graph"] = F.ApplyGraph(V, lam, f, pf, pa, pair_t=state["pt"], ctx=ctx)
        return state
    if kind == "solve":
        mask = _mask(case["dim"], case["grid"], case["n"], seed)
        pf, pa = _pairs(case["m"], case["orders"], seed)
        mixed = case["route"] == "mixed"
        return {"kind": kind, "mixed": mixed, "ctx": _context(64, 6) if mixed else _context(), "h": 1.0 / (case["grid"] + 1),
                "mask": torch.from_numpy(mask).cuda(), "F": _forcings(mask, case["m"], seed), "pf": pf, "pa": pa}
    if kind == "batch":
        items = []
        for i, side in enumerate(_sides(case)):
            mask = _mask(2, side, 9 * side * side // 20, 1000 * seed + i)
            pf, pa = _pairs(case["m"], case["orders"], 1000 * seed + i)
            items.append({"mask": torch.from_numpy(mask).cuda(), "h": 1.0 / (side + 1), "F": _forcings(mask, case["m"], 1000 * seed + i),
                          "pair_f": pf.cpu().numpy(), "pair_alpha": pa.cpu().numpy()})
        return {"kind": kind, "ctx": _context(), "items": items}
    if kind == "fem":
        mask = _mask(2, case["grid"], case["n"], seed)
        pf, pa = _pairs(case["m"], case["orders"], seed)
        return {"kind": kind, "ctx": _context(), "h": 1.0 / (case["grid"] + 1), "mask": torch.from_numpy(mask).cuda(),
                "F": _forcings(mask, case["m"], seed), "pf": pf, "pa": pa}
    if kind == "product":
        A, B = _product_inputs(case, seed)
        return {"kind": kind, "ctx": _context(), "A": A, "B": B, "slices": case["slices"]}
    h = 1.0 / (case["grid"] + 1)
    asm = F.fd_assemble(torch.from_numpy(_mask(2, case["grid"], case["n"], seed)).cuda(), h, dense=False, ctx=_context())
    sigmas = np.sort(np.random.default_rng([seed, 13]).uniform(0.0, 8.0 / h ** 2, size=case["shifts"]))
    return {"kind": kind, "ctx": _context(), "csr": (asm["rowptr"], asm["col"], asm["val"]), "sigmas": torch.from_numpy(sigmas).cuda(),
            "band": F.csr_half_bandwidth(asm["rowptr"], asm["col"], ctx=_context())}


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------
def run(state):
    kind, ctx = state["kind"], state["ctx"]
    if kind == "apply":
        if state["graph"] is not None:
            return state["graph"].launch(sync=False)
        if state["pt"] is not None:
            return F.frac_diffusion(state["V"], state["lam"], state["F"], state["pf"], state["pa"], state["pt"], mu=1.0, ctx=ctx, sync=False)
        return F.frac_apply(state["V"], state["lam"], state["F"], state["pf"], state["pa"], ctx=ctx, sync=False)
    if kind == "solve":
        if not state["mixed"]:
            lam, _, U = F.solve(state["mask"], state["h"], state["F"], state["pf"], state["pa"], ctx=ctx)
            return {"lambda": lam, "U": U}
        asm = F.fd_assemble(state["mask"], state["h"], ctx=ctx)
        lam, V = F.eig_full_mixed(asm["A"], asm["rowptr"], asm["col"], asm["val"], refine_iters=6, ctx=ctx)
        return {"lambda": lam, "U": F.frac_apply(V, lam, state["F"], state["pf"], state["pa"], ctx=ctx)}
    if kind == "batch":
        problems = []
        for it in state["items"]:
            asm = F.fd_assemble(it["mask"], it["h"], ctx=ctx)
            problems.append({"A": asm["A"], "rowptr": asm["rowptr"], "col": asm["col"], "val": asm["val"], "F": it["F"],
                             "pair_f": it["pair_f"], "pair_alpha": it["pair_alpha"]})
        # one vector each over all problems: there are more problems than outputs a caller would list
        out = F.solve_batched(problems, ctx=ctx)
        return {"lambda": torch.cat([lam for lam, _, _ in out]), "U": torch.cat([U.t().reshape(-1) for _, _, U in out])}
    if kind == "fem":
        fem = F.fem_assemble(state["mask"], state["h"], ctx=ctx)
        theta, Phi = F.eig_pencil(fem["K"], fem["rowptr"], fem["col"], fem["valM"], ctx=ctx)
        U = F.frac_apply_mass(Phi, theta, fem["rowptr"], fem["col"], fem["valM"], state["F"], state["pf"], state["pa"], ctx=ctx)
        return {"theta": theta, "U": U}
    if kind == "product":
        return F.dgemm_ozaki(state["A"], state["B"], trans_a=True, slices=state["slices"], ctx=ctx)
    return F.inertia_counts(*state["csr"], state["sigmas"], half_bandwidth=state["band"], ctx=ctx, sync=False)


# ----------------------------------------------------------------------------
# what a pass cannot do without, and what it should return
# ----------------------------------------------------------------------------
def _eig_flops(n):
    # tridiagonal reduction 4/3, eigenvectors of the tridiagonal matrix 4/3, one back-transformation 2
    return (4.0 / 3.0 + 4.0 / 3.0 + 2.0) * n ** 3


def work(case):
    kind = case["kind"]
    if kind == "apply":
        n, m, k = case["nx"] * case["ny"], case["m"], case["k"]
        return {"bytes": 8.0 * (n * n + n + n * m + n * k) + 12.0 * k, "flops": 2.0 * n * n * (m + k)}
    if kind in ("solve", "fem"):
        n, m, k = case["n"], case["m"], case["m"] * case["orders"]
        return {"bytes": 8.0 * (2 * n * n + n + n * m + n * k), "flops": _eig_flops(n) + 2.0 * n * n * (m + k)}
    if kind == "batch":
        m, k, w = case["m"], case["m"] * case["orders"], {"bytes": 0.0, "flops": 0.0}
        for n in (9 * side * side // 20 for side in _sides(case)):
            w["bytes"] += 8.0 * (2 * n * n + n + n * m + n * k)
            w["flops"] += _eig_flops(n) + 2.0 * n * n * (m + k)
        return w
    if kind == "product":
        r, c, i = case["rows"], case["cols"], case["inner"]
        return {"bytes": 8.0 * (r * i + c * i + r * c), "flops": 2.0 * r * c * i}
    # one banded LDL^T per shift, band of about the grid's row length
    return {"bytes": 12.0 * 5 * case["n"] + 16.0 * case["shifts"], "flops": 1.0 * case["shifts"] * case["n"] * case["grid"] ** 2}


def _laplacian(mask, h):
    """Dense 5- / 7-point Dirichlet Laplacian of the mask, on the GPU."""
    keep = torch.from_numpy(mask.astype(bool)).cuda()
    n = int(keep.sum())
    idx = torch.full(mask.shape, -1, dtype=torch.int64, device="cuda")
    idx[keep] = torch.arange(n, device="cuda")
    A = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    A.fill_diagonal_(2.0 * mask.ndim / (h * h))
    for d in range(mask.ndim):
        a, b = idx.narrow(d, 0, mask.shape[d] - 1), idx.narrow(d, 1, mask.shape[d] - 1)
        both = (a >= 0) & (b >= 0)
        A[a[both], b[both]] = A[b[both], a[both]] = -1.0 / (h * h)
    return A


def _fem(mask, h):
    """Dense bilinear stiffness and mass matrices of the mask: sums of tensor products of the 1-D ones."""
    c = mask.shape[0]
    eye, off = torch.eye(c, dtype=torch.float64, device="cuda"), torch.zeros(c, c, dtype=torch.float64, device="cuda")
    i = torch.arange(c - 1, device="cuda")
    off[i, i + 1] = off[i + 1, i] = 1.0
    k1, m1 = (2 * eye - off) / h, (4 * eye + off) * (h / 6)
    keep = torch.from_numpy(np.flatnonzero(mask.reshape(-1))).cuda()
    cut = lambda a: a[keep][:, keep]  # noqa: E731
    return cut(torch.kron(m1, k1) + torch.kron(k1, m1)), cut(torch.kron(m1, m1))


def _spectral(lam, V, coeffs, pf, pa):
    return V @ (coeffs[:, pf.long()] * lam[:, None] ** (-pa[None, :] / 2))


def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":
        lam, V, f, pf, pa, pt = _apply_inputs(case, seed)
        w = (V.t() @ f)[:, pf.long()]
        scale = torch.exp(-lam[:, None] ** (pa[None, :] / 2) * pt[None, :]) if case["times"] else lam[:, None] ** (-pa[None, :] / 2)
        return V @ (w * scale)
    if kind == "solve":
        mask = _mask(case["dim"], case["grid"], case["n"], seed)
        pf, pa = _pairs(case["m"], case["orders"], seed)
        lam, V = torch.linalg.eigh(_laplacian(mask, 1.0 / (case["grid"] + 1)))
        return {"lambda": lam, "U": _spectral(lam, V, V.t() @ _forcings(mask, case["m"], seed), pf, pa)}
    if kind == "batch":
        lams, us = [], []
        for i, side in enumerate(_sides(case)):
            mask = _mask(2, side, 9 * side * side // 20, 1000 * seed + i)
            pf, pa = _pairs(case["m"], case["orders"], 1000 * seed + i)
            lam, V = torch.linalg.eigh(_laplacian(mask, 1.0 / (side + 1)))
            lams.append(lam)
            us.append(_spectral(lam, V, V.t() @ _forcings(mask, case["m"], 1000 * seed + i), pf, pa).t().reshape(-1))
        return {"lambda": torch.cat(lams), "U": torch.cat(us)}
    if kind == "fem":
        mask = _mask(2, case["grid"], case["n"], seed)
        pf, pa = _pairs(case["m"], case["orders"], seed)
        K, M = _fem(mask, 1.0 / (case["grid"] + 1))
        L = torch.linalg.cholesky(M)
        half = torch.linalg.solve_triangular(L, K, upper=False)
        C = torch.linalg.solve_triangular(L, half.t(), upper=False)
        theta, Z = torch.linalg.eigh((C + C.t()) / 2)
        Phi = torch.linalg.solve_triangular(L.t(), Z, upper=True)
        return {"theta": theta, "U": _spectral(theta, Phi, Phi.t() @ (M @ _forcings(mask, case["m"], seed)), pf, pa)}
    if kind == "product":
        A, B = _product_inputs(case, seed)
        return A.t() @ B
    return None  # whole numbers
