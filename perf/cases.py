"""The work that the solver's speed is judged by: cases over the range of sizes, fields and options in use.

A case is one call that a reservoir or inversion code makes: a PCG solve with a prepared handle, a
batch of right-hand sides with their adjoints, a block solve, or one evaluation of the
differentiable pressure solve (assembly, setup, forward and adjoint solve, gradient).  The inputs
are seeded draws on the GPU of the synthetic fields in ``paper_1205_6113_gb300.inputs``: an iid
lognormal plane, a Gaussian-correlated field and sinuous high-permeability channels.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1205_6113_gb300 import adjoint, cpc, inputs

DEV = "cuda"
#: Anisotropy k_z / k of each field, as in the generators of the package.
KZ = {"lognormal": 1.0, "correlated": 0.1, "channels": 0.01}


def _solve(name, field, nx, ny, nz, precond="bco", precision="fp64", ic_order="colour", gs_order="multicolour",
           system="tpfa", tol=1e-6):
    return dict(name=name, kind="solve", system=system, field=field, nx=nx, ny=ny, nz=nz, precond=precond,
                precision=precision, ic_order=ic_order, gs_order=gs_order, tol=tol)


def listed():
    return [
        # The plane of the plain method: a call so small that latency and launches are all there is.
        _solve("plane_64x64", "lognormal", 64, 64, 1),
        # Solver() as it comes: natural-order IC(0) inside B_co, at the paper's tolerance, on a ragged grid.
        _solve("default_61x53x37", "correlated", 61, 53, 37, ic_order="natural", tol=1e-10),
        # The benchmark's field: one million cells, all FP64 and with the FP32 preconditioner.
        _solve("field_1m_fp64", "correlated", 128, 128, 64),
        _solve("field_1m_fp32", "correlated", 128, 128, 64, precision="fp32"),
        # AMG alone with BF16 coarse operators on a ragged channel field: the least memory an operator takes.
        _solve("amg_bf16_101x87x45", "channels", 101, 87, 45, precond="amg", precision="fp32_bf16"),
        # The largest model: 8.4 million cells, a 1000:1 channel field, FP64.
        _solve("channels_8m_fp64", "channels", 256, 256, 128),
        # Mixed-hybrid (p, lambda) system: 530 thousand unknowns, no structured fine level, positive couplings.
        _solve("mhfem_64x64x32", "channels", 64, 64, 32, system="mhfem"),
        # IC(0) alone in its natural order: the baseline that the paper compares with, on a small model.
        _solve("ic0_40x36x20", "correlated", 40, 36, 20, precond="ic0", ic_order="natural"),
        # 64 well patterns and their adjoints on the benchmark's field, FP32 preconditioner.
        dict(name="adjoints_1m_k64", kind="adjoints", field="correlated", nx=128, ny=128, nz=64, columns=64,
             precision="fp32", tol=1e-6),
        # A ragged handful of coupled right-hand sides by block CG, FP64.
        dict(name="block_80x72x30_k12", kind="block", field="correlated", nx=80, ny=72, nz=30, columns=12,
             precision="fp64", tol=1e-6),
        # One gradient of a well misfit, as each step of an inversion asks for: log k is new each time, so
        # assembly and setup are part of the call.
        dict(name="gradient_96x80x48", kind="gradient", field="channels", nx=96, ny=80, nz=48, tol=1e-8),
    ]


def _grid(rng, lo, hi, flat):
    """A ragged grid of about n cells, n log-uniform in [lo, hi]: a plane when flat."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if flat:
        a = math.exp(rng.uniform(-0.7, 0.7))
        nx = max(8, round(math.sqrt(n) * a))
        return nx, max(8, int(n / nx)), 1
    a, b = math.exp(rng.uniform(-0.4, 0.4)), math.exp(rng.uniform(-1.0, 0.0))
    side = (n / b) ** (1.0 / 3.0)
    nx = max(8, round(side * a))
    nz = max(4, round(side * b))
    return nx, max(8, int(n / (nx * nz))), nz


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["adjoints", "block", "gradient"])
    field = rng.choice(["lognormal", "correlated", "channels"])
    tol = rng.choice([1e-6, 1e-6, 1e-8, 1e-10])
    if kind == "solve":
        system = "mhfem" if field != "lognormal" and rng.random() < 0.15 else "tpfa"
        precond = rng.choice(["bco"] * 5 + ["amg"] * 2 + ["ic0", "bhat", "amg_ilu"] * (system == "tpfa"))
        ic_order = rng.choice(["colour", "colour", "natural"])
        gs_order = "natural" if ic_order == "natural" and rng.random() < 0.2 else "multicolour"
        hi = 8.0e6                                    # IC(0) alone and natural sweeps take far longer per cell
        if field == "lognormal" or system == "mhfem":
            hi = 1.0e6
        if ic_order == "natural":
            hi = 5.0e5
        if precond == "ic0" or gs_order == "natural":
            hi = 5.0e4
        nx, ny, nz = _grid(rng, 2.0e3, hi, field == "lognormal")
        precision = rng.choice(["fp64", "fp64", "fp32", "fp32_bf16"])
        c = _solve("", field, nx, ny, nz, precond, precision, ic_order, gs_order, system, tol)
        del c["name"]
        return c
    if kind == "gradient":
        nx, ny, nz = _grid(rng, 2.0e3, 1.0e6, field == "lognormal")
        return dict(kind=kind, field=field, nx=nx, ny=ny, nz=nz, tol=min(tol, 1e-8))
    columns = rng.randint(1, 128 if kind == "adjoints" else 64)
    nx, ny, nz = _grid(rng, 2.0e3, min(1.0e6, 3.2e7 / columns), field == "lognormal")
    return dict(kind=kind, field=field, nx=nx, ny=ny, nz=nz, columns=columns,
                precision=rng.choice(["fp64", "fp32", "fp32_bf16"]) if kind == "adjoints" else "fp64", tol=1e-6)


# -- inputs --------------------------------------------------------------------------------------


def _logk(case, seed):
    """log k on the GPU, flat in natural order (x fastest)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    if case["field"] == "lognormal":
        return torch.randn(nx * ny * nz, generator=gen, device=DEV, dtype=torch.float64)
    if case["field"] == "correlated":
        noise = torch.randn((nz, ny, nx), generator=gen, device=DEV, dtype=torch.float64)
        r2 = 0.0
        for d, s in enumerate((nz, ny, nx)):
            i = torch.arange(s, device=DEV, dtype=torch.float64)
            shape = [1, 1, 1]
            shape[d] = s
            r2 = r2 + torch.minimum(i, s - i).square().reshape(shape)
        f = torch.fft.ifftn(torch.fft.fftn(noise) * torch.fft.fftn(torch.exp(-2.0 * r2 / 64.0))).real
        return (2.0 * (f - f.mean()) / f.std()).reshape(-1).contiguous()
    # channels: y = y0 + a sin(2 pi x / lam + phi), 12 cells wide and 6 layers thick, to a quarter of the volume
    rng = np.random.default_rng(seed)
    facies = np.zeros((nz, ny, nx), dtype=bool)
    xs, ys = np.arange(nx), np.arange(ny)
    while facies.mean() < 0.25:
        for _ in range(max(1, nz // 16)):
            a, lam, phi = rng.uniform(8.0, 32.0), rng.uniform(64.0, 256.0), rng.uniform(0.0, 2.0 * np.pi)
            y0, z0 = rng.uniform(0.0, ny), int(rng.integers(0, max(1, nz - 5)))
            yc = y0 + a * np.sin(2.0 * np.pi * xs / lam + phi)
            facies[z0:z0 + 6] |= (np.abs(ys[:, None] - yc[None, :]) < 6.0)[None]
    return torch.from_numpy(facies.reshape(-1)).to(DEV).double() * math.log(1000.0)


def _problem(case):
    p = inputs.Problem("case", case["nx"], case["ny"], case["nz"], None, KZ[case["field"]], inputs.FACE_X0)
    if case["field"] == "lognormal":
        p.wells = [(p.idx(3 * p.nx // 4, 3 * p.ny // 4), 1.0)]
    elif case["field"] == "correlated":
        p.wells = inputs.five_spot(p, p.nz // 2)
    else:
        p.wells = inputs.nine_wells(p)
    return p


def _matrix(case, p, logk):
    assemble = cpc.mhfem_assemble if case.get("system") == "mhfem" else cpc.tpfa_assemble
    return assemble(p.nx, p.ny, p.nz, logk, p.kz_ratio, p.dirichlet)


def _rhs(p, n, seed):
    """Well rates, each within 20% of the pattern's own."""
    rng = np.random.default_rng(seed + 1)
    cells = torch.tensor([c for c, _ in p.wells], device=DEV)
    rates = torch.tensor([q * rng.uniform(0.8, 1.2) for _, q in p.wells], device=DEV, dtype=torch.float64)
    b = torch.zeros(n, device=DEV, dtype=torch.float64)
    return b.index_put_((cells,), rates, accumulate=True)


def _columns(n, columns, seed):
    """[n, columns] right-hand sides, each with rates U[-1, 1] at 16 random cells."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed + 1)
    B = torch.zeros(n, columns, device=DEV, dtype=torch.float64)
    cells = torch.randint(n, (16, columns), generator=gen, device=DEV)
    return B.scatter_(0, cells, 2.0 * torch.rand(16, columns, generator=gen, device=DEV, dtype=torch.float64) - 1.0)


def _wells(p):
    """Well cells and the pressures observed in them."""
    cells = torch.tensor(inputs.well_columns(p), device=DEV)
    observed = torch.linspace(-1.0, 1.0, cells.shape[0], device=DEV, dtype=torch.float64)
    return cells, observed


def prepare(case, seed):
    p = _problem(case)
    logk = _logk(case, seed)
    state = dict(case=case, p=p)
    if case["kind"] == "gradient":
        cells, observed = _wells(p)
        return dict(state, logk=logk.requires_grad_(), q=_rhs(p, p.n, seed).requires_grad_(), cells=cells,
                    observed=observed)
    rowptr, col, val = _matrix(case, p, logk)
    n = rowptr.shape[0] - 1
    if case["kind"] == "solve":
        solver = cpc.Solver(rowptr, col, val, precond=case["precond"], precision=case["precision"],
                            ic_order=case["ic_order"], gs_order=case["gs_order"])
        return dict(state, solver=solver, b=_rhs(p, n, seed))
    solver = cpc.Solver(rowptr, col, val, precision=case["precision"], ic_order="colour")
    return dict(state, solver=solver, B=_columns(n, case["columns"], seed))


def run(state):
    case = state["case"]
    if case["kind"] == "solve":
        x, iters, status, _ = state["solver"].solve(state["b"], tol=case["tol"], maxit=5000, hist=False)
        return dict(x=x, iters=iters, status=status)
    if case["kind"] == "adjoints":
        X, Lam, itf, ita = state["solver"].solve_batched_adjoint(state["B"], tol=case["tol"])
        return dict(x=X, adjoint=Lam, iters=itf, iters_adjoint=ita)
    if case["kind"] == "block":
        X, iters, _, status = state["solver"].solve_block(state["B"], tol=case["tol"])
        return dict(x=X, iters=iters, status=status)
    p = state["p"]
    grid = adjoint.Grid(p.nx, p.ny, p.nz, p.kz_ratio, p.dirichlet)
    pres = adjoint.pressure(state["logk"], state["q"], grid, tol=case["tol"])
    misfit = 0.5 * (adjoint.well_pressures(pres, state["cells"]) - state["observed"]).square().sum()
    g_logk, g_q = torch.autograd.grad(misfit, (state["logk"], state["q"]))
    return dict(x=pres.detach(), g_logk=g_logk, g_q=g_q)


def _sizes(case):
    """(unknowns, nonzeros) of the case's matrix."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = nx * ny * nz
    faces = (nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1)
    if case.get("system") != "mhfem":
        return n, n + 2 * faces
    free = faces + ny * nz + 2 * nx * nz + 2 * nx * ny       # every face but those of x = 0
    return n + free, n + 2 * (6 * n - ny * nz) + free + 6 * n - 2 * ny * nz


def work(case):
    """The matrix read once, the right-hand sides read and the results written once; as operations, a
    sweep, a residual and a product with the matrix in each of ten iterations."""
    n, nnz = _sizes(case)
    k = case.get("columns", 1)
    passes = 2 if case["kind"] in ("adjoints", "gradient") else 1
    vectors = {"solve": 2, "block": 2, "adjoints": 3, "gradient": 5}[case["kind"]]
    matrix = 0 if case["kind"] == "gradient" else 12 * nnz + 4 * (n + 1)
    return {"bytes": matrix + 8 * vectors * n * k, "flops": 10 * passes * 3 * 2 * nnz * k}


# -- 64-bit results from torch alone ---------------------------------------------------------------


def _faces(case, kz):
    """For each axis: the flat indices of the cells on either side of its inner faces, and k_f / k."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    c = torch.arange(nx * ny * nz, device=DEV).reshape(nz, ny, nx)
    return [(c[:, :, :-1].reshape(-1), c[:, :, 1:].reshape(-1), 1.0),
            (c[:, :-1, :].reshape(-1), c[:, 1:, :].reshape(-1), 1.0),
            (c[:-1].reshape(-1), c[1:].reshape(-1), kz)]


def _csr(n, rows, cols, vals):
    a = torch.sparse_coo_tensor(torch.stack([torch.cat(rows), torch.cat(cols)]), torch.cat(vals), (n, n)).coalesce()
    diag = torch.zeros(n, device=DEV, dtype=torch.float64)
    i, v = a.indices(), a.values()
    on = i[0] == i[1]
    diag[i[0][on]] = v[on]
    return a.to_sparse_csr(), diag


def _tpfa(case, logk):
    p = _problem(case)
    k, rows, cols, vals = torch.exp(logk), [], [], []
    for a, b, s in _faces(case, p.kz_ratio):
        t = 2.0 * s * k[a] * k[b] / (k[a] + k[b])
        rows += [a, b, a, b]
        cols += [b, a, a, b]
        vals += [-t, -t, t, t]
    x0 = torch.arange(0, p.n, p.nx, device=DEV)
    return _csr(p.n, rows + [x0], cols + [x0], vals + [2.0 * k[x0]])


def _mhfem(case, logk):
    """Cells, then the free x-, y- and z-faces in (k, j, i) order; the faces of x = 0 are held at 0."""
    p = _problem(case)
    nx, ny, nz = p.nx, p.ny, p.nz
    k = torch.exp(logk)
    cell = torch.arange(p.n, device=DEV)
    i, j, l = cell % nx, cell // nx % ny, cell // (nx * ny)
    fx, fy = nx * ny * nz, nx * (ny + 1) * nz
    pairs = [(torch.where(i > 0, i - 1 + nx * (j + ny * l), -1), i + nx * (j + ny * l), 1.0),
             (fx + i + nx * (j + (ny + 1) * l), fx + i + nx * (j + 1 + (ny + 1) * l), 1.0),
             (fx + fy + i + nx * (j + ny * l), fx + fy + i + nx * (j + ny * (l + 1)), p.kz_ratio)]
    rows, cols, vals = [], [], []

    def add(r, c, v):
        ok = (r >= 0) & (c >= 0)
        rows.append(r[ok])
        cols.append(c[ok])
        vals.append(v[ok])

    for lo, hi, s in pairs:
        f = s * k
        add(cell, cell, 12.0 * f)
        lo, hi = torch.where(lo >= 0, lo + p.n, -1), hi + p.n
        for u, v in ((lo, hi), (hi, lo)):
            add(cell, u, -6.0 * f)
            add(u, cell, -6.0 * f)
            add(u, u, 4.0 * f)
            add(u, v, 2.0 * f)
    return _csr(p.n + fx + fy + nx * ny * (nz + 1), rows, cols, vals)


def _cg(A, diag, B):
    """Jacobi-preconditioned CG on the columns of B to a relative residual of 1e-13, or None."""
    X, R = torch.zeros_like(B), B.clone()
    d = diag[:, None]
    norm = B.norm(dim=0)
    norm[norm == 0] = 1.0
    P = R / d
    rz = (R * P).sum(0)
    for it in range(20000):
        Q = A @ P
        pq = (P * Q).sum(0)
        alpha = torch.where(pq > 0, rz / pq, 0.0)
        X += alpha * P
        R -= alpha * Q
        Z = R / d
        new = (R * Z).sum(0)
        P = Z + torch.where(rz > 0, new / rz, 0.0) * P
        rz = new
        if it % 100 == 99 and bool((R.norm(dim=0) < 1e-13 * norm).all()):
            return X
    return None


def exact(case, seed):
    n, _ = _sizes(case)
    if n * case.get("columns", 1) > 2_500_000:        # thousands of iterations: more than 20 seconds
        return None
    p = _problem(case)
    logk = _logk(case, seed)
    A, diag = (_mhfem if case.get("system") == "mhfem" else _tpfa)(case, logk)
    if case["kind"] in ("adjoints", "block"):
        B = _columns(n, case["columns"], seed)
        X = _cg(A, diag, B)
        if case["kind"] == "block":
            return None if X is None else dict(x=X, iters=None, status=None)
        L = None if X is None else _cg(A, diag, torch.where(B != 0, X, 0.0))
        return None if L is None else dict(x=X, adjoint=L, iters=None, iters_adjoint=None)
    b = _rhs(p, n, seed)
    X = _cg(A, diag, b[:, None])
    if X is None:
        return None
    x = X[:, 0]
    if case["kind"] == "solve":
        return dict(x=x, iters=None, status=None)
    cells, observed = _wells(p)
    dj = torch.zeros(n, device=DEV, dtype=torch.float64)
    miss = (x[cells].mean(dim=1) - observed) / cells.shape[1]
    dj.index_put_((cells.reshape(-1),), miss.repeat_interleave(cells.shape[1]), accumulate=True)
    L = _cg(A, diag, dj[:, None])
    if L is None:
        return None
    lam, k, g = L[:, 0], torch.exp(logk), torch.zeros(n, device=DEV, dtype=torch.float64)
    for a, c, s in _faces(case, p.kz_ratio):          # -lambda^T (dA / dlog k) x, face by face
        jump = s * (lam[a] - lam[c]) * (x[a] - x[c])
        g.index_add_(0, a, -2.0 * k[a] * (k[c] / (k[a] + k[c])) ** 2 * jump)
        g.index_add_(0, c, -2.0 * k[c] * (k[a] / (k[a] + k[c])) ** 2 * jump)
    x0 = torch.arange(0, n, p.nx, device=DEV)
    g[x0] -= 2.0 * k[x0] * lam[x0] * x[x0]
    return dict(x=x, g_logk=g, g_q=lam)
