"""Sweeps and triangular solves that run as one launch ordered by their data, and the sweeps by colour
launches from a zero guess: every row of every level satisfies its own equation, to rounding.

A row of a forward sweep from zero solves (D + L) y = x, of a backward sweep (D + U) y = x, of a forward
sweep from y0 (D + L) y + U y0 = x, with L and U the couplings to earlier and later colours.  A sum of m
products computed in any order, a difference and a product with the stored reciprocal of a_ii leave a
residual of at most (m + 4) eps times the sum of the magnitudes of the row's terms.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_1205_6113_gb300 import cpc, inputs  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
EPS = np.finfo(np.float64).eps


def solver(p, **kw):
    csr = cpc.tpfa_assemble(p.nx, p.ny, p.nz, torch.tensor(p.logk, device=DEV), p.kz_ratio, p.dirichlet)
    return cpc.Solver(*csr, **kw)


def worst(s, l, y, x, y0, forward):
    """max over the rows of level l of |residual| / ((m + 4) eps sum of magnitudes)."""
    ptr, col, val = s.level_matrix(l)
    _, colour = s.level_splitting(l)
    n = ptr.size - 1
    rows = np.repeat(np.arange(n), np.diff(ptr))
    earlier = colour[col] < colour[rows]
    new = (rows == col) | (earlier if forward else colour[col] > colour[rows])
    t = val * np.where(new, y[col], y0[col])
    res = np.bincount(rows, weights=t, minlength=n) - x
    mag = np.bincount(rows, weights=np.abs(t), minlength=n) + np.abs(x)
    return float(np.max(np.abs(res) / ((np.diff(ptr) + 4) * EPS * mag)))


# one colour and one row left over; few chunks per colour; blocks of four warps; colour launches on level 1
@pytest.mark.parametrize("shape,kw", [((33, 1, 1), dict(coarse_max=8)), ((13, 11, 7), dict(coarse_max=16)),
                                      ((13, 11, 7), dict(coarse_max=16, gs_order="natural")), ((61, 53, 37), {}),
                                      ((101, 87, 45), {}), ((128, 128, 64), {})])
def test_every_row_solves_its_equation(shape, kw):
    s = solver(inputs.small_3d(*shape, seed=81), **kw)
    for l in range(s.nlevels - 1):
        n = s.level_info(l)["n"]
        x, y0 = inputs.random_vector(n, 82 + l), inputs.random_vector(n, 92 + l)
        xd, zero = torch.tensor(x, device=DEV), np.zeros(n)
        assert worst(s, l, s.level_apply(l, 1, xd).cpu().numpy(), x, zero, True) <= 1.0
        assert worst(s, l, s.level_apply(l, 2, xd).cpu().numpy(), x, zero, False) <= 1.0
        y = s.level_apply(l, 5, xd, torch.tensor(y0, device=DEV)).cpu().numpy()
        assert worst(s, l, y, x, y0, True) <= 1.0


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_bf16"])
@pytest.mark.parametrize("which", ["bco", "ic0", "amg_ilu"])
def test_applications_repeat_to_the_bit(which, precision):
    """Sums are taken in entry order whatever the order of arrival; and a NaN on one row spreads, it
    does not hang or turn into a number."""
    p = inputs.small_3d(40, 36, 20, seed=83)
    s = solver(p, precond=which, precision=precision)
    r = torch.tensor(inputs.random_vector(p.n, 84), device=DEV)
    z = s.apply(r)
    for _ in range(5):
        assert torch.equal(s.apply(r), z)
    bad = r.clone()
    bad[p.n // 2] = float("nan")
    assert bool(torch.isnan(s.apply(bad)).any())
    assert torch.equal(s.apply(r), z)


def test_in_place_ic0():
    """z = r as one buffer: every row is read before it is written."""
    p = inputs.small_3d(40, 36, 20, seed=85)
    s = solver(p, precond="ic0")
    r = torch.tensor(inputs.random_vector(p.n, 86), device=DEV)
    z = s.apply(r)
    buf = r.clone()
    assert torch.equal(s.apply(buf, z=buf), z)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("K", [1, 8, 9, 16, 17, 33, 64, 65, 96, 97, 128])
def test_batched_paddings_repeat_single_solves(K, precision):
    """Every width that block vectors are padded to (8, 16, multiples of 32), at its edges: each column
    takes the iterations of its own single solve and agrees with it.  The two differ by the rounding of
    their sums alone, a relative 1e-15 in FP64 and 1e-6 in FP32 of the iteration error, which ends
    below 1e-6; the bound leaves a factor of 1000 for its growth along the recurrences."""
    p = inputs.small_3d(21, 19, 11, seed=87)
    s = solver(p, coarse_max=64, ic_order="colour", precision=precision)
    B = torch.tensor(np.ascontiguousarray(inputs.batch_rhs(p.n, K, cells_per_rhs=4, seed=88).T), device=DEV)
    bound = 1e-12 if precision == "fp64" else 1e-9
    for _ in range(2):                                   # the second call replays the graph on other buffers
        X, it, st = s.solve_batched(B, tol=1e-6, maxit=100)
        assert not st.any()
        for k in sorted({0, K // 2, K - 1}):
            x, iters, status, _ = s.solve(B[:, k].contiguous(), tol=1e-6, maxit=100)
            assert status == 0 and iters == it[k]
            assert float((X[:, k] - x).norm() / x.norm()) <= bound


# one row per lane group and a few left over; a full batch of four rows and one left over
@pytest.mark.parametrize("shape", [(19, 16, 16), (33, 33, 18)])
@pytest.mark.parametrize("K,precision", [(8, "fp64"), (16, "fp32"), (31, "fp32"), (33, "fp32"), (64, "fp64"), (90, "fp32"), (128, "fp32")])
def test_batched_rows_left_over(shape, K, precision):
    """Every column reaches the tolerance in its true residual (which differs from the recurrence's by
    rounding, far less than the tolerance), in as many iterations as its own solve to one."""
    p = inputs.small_3d(*shape, seed=85)
    csr = cpc.tpfa_assemble(p.nx, p.ny, p.nz, torch.tensor(p.logk, device=DEV), p.kz_ratio, p.dirichlet)
    s = cpc.Solver(*csr, precision=precision, ic_order="colour")
    n = p.nx * p.ny * p.nz
    B = torch.tensor(inputs.random_vector(n * K, 86).reshape(n, K), device=DEV)
    X, it, st = s.solve_batched(B, tol=1e-8, maxit=500)
    assert np.all(st == 0)
    A = torch.sparse_csr_tensor(*csr, size=(n, n))
    res = (torch.linalg.vector_norm(B - A @ X, dim=0) / torch.linalg.vector_norm(B, dim=0)).cpu().numpy()
    assert np.all(res <= 2e-8)
    for k in (0, K // 2, K - 1):
        _, its, sts, _ = s.solve(B[:, k].contiguous(), tol=1e-8, maxit=500)
        assert sts == 0 and abs(int(it[k]) - its) <= 1


def test_wide_ic0_levels_keep_their_launches():
    """IC(0) of a mixed-hybrid system in its four colours, 258,000 rows each: a launch per level and factor,
    where the natural order's narrow levels take one per factor.  The solve of L (U z) = r, rows of at
    most m products, leaves a residual of at most 2 (m + 5) eps (|L| |U| |z| + |r|) per row."""
    import scipy.sparse as sp
    nx, ny, nz = 80, 80, 40
    logk = torch.tensor(inputs.random_vector(nx * ny * nz, 89), device=DEV)
    csr = cpc.mhfem_assemble(nx, ny, nz, logk, 0.1, inputs.FACE_X0)
    s = cpc.Solver(*csr, precond="ic0", ic_order="colour")
    t = cpc.Solver(*csr, precond="ic0")
    levels = s.level_info(0)["ic_levels"]
    assert 2 < levels and s.n // levels > 200000 > t.n // t.level_info(0)["ic_levels"]
    assert s.solve_launches()[0] == t.solve_launches()[0] - 2 + 2 * levels
    r = inputs.random_vector(s.n, 90)
    z = s.apply(torch.tensor(r, device=DEV)).cpu().numpy()
    ptr, col, val = (a.cpu().numpy() for a in csr)
    order = np.argsort(s.level_splitting(0)[1], kind="stable")
    F = sp.csr_matrix((val, col, ptr), shape=(s.n, s.n))[order][:, order]
    F.sort_indices()
    F.data = s.ic0_values()
    L, U = sp.tril(F, -1) + sp.identity(s.n), sp.triu(F)
    r, z = r[order], z[order]
    bound = 2 * (np.diff(F.indptr).max() + 5) * EPS * (abs(L) @ (abs(U) @ abs(z)) + abs(r))
    assert np.all(np.abs(L @ (U @ z) - r) <= bound)


def test_sweeps_of_more_chunks_than_the_gpu_holds_keep_their_launches():
    """Level 2 of 5 million cells in FP32, 18,000 rows a colour in chunks of 8 rows: more than three quarters of
    the 2,432 warps that the GPU holds of a sweep with 16 entries to a lane.  An iteration has five kernels
    of the loop and two cycles of at least 7 launches on the red-black level 0, on levels 1 and 2 of g colours
    g - 1 forward from zero (the first colour comes with the restriction), g backward and 3 for residual and
    transfers, and the coarsest solve."""
    nx, ny, nz = 216, 216, 108
    gen = torch.Generator(device=DEV)
    gen.manual_seed(91)
    logk = torch.randn(nx * ny * nz, generator=gen, device=DEV, dtype=torch.float64)
    s = cpc.Solver(*cpc.tpfa_assemble(nx, ny, nz, logk, 0.1, inputs.FACE_X0), precond="amg", precision="fp32")
    i = s.level_info(2)
    assert i["n"] // i["ncolours"] <= 24000 and i["n"] / (s.level_layout(2)["C"] * i["ncolours"]) > 0.75 * 2432
    by_colours = sum(2 * s.level_info(l)["ncolours"] - 1 + 3 for l in (1, 2))
    assert s.solve_launches()[0] >= 5 + 2 * (7 + by_colours + 1)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_a_wait_that_gives_up_is_reported_once(precision):
    """With one poll a wait, rows of later wavefronts give up at once (the first of them start together): the
    launches end, the result holds NaN, the next call that synchronises says so, and nothing is left behind."""
    p = inputs.small_3d(40, 36, 20, seed=92)
    s = solver(p, precision=precision)
    b = torch.tensor(inputs.random_vector(p.n, 93), device=DEV)
    z = s.apply(b)
    x, iters, status, _ = s.solve(b, tol=1e-8)
    for call in (lambda: s.solve(b, tol=1e-8), lambda: s.sweep_time_us(1)):
        s.set_wait_polls(1)
        assert bool(torch.isnan(s.apply(b)).any())
        s.set_wait_polls(0)
        with pytest.raises(cpc.CpcError) as e:
            call()
        assert e.value.code == 6
        assert torch.equal(s.apply(b), z)
        again = s.solve(b, tol=1e-8)
        assert torch.equal(again[0], x) and again[1:3] == (iters, status)
    s.set_wait_polls(1)
    with pytest.raises(cpc.CpcError) as e:
        s.solve(b, tol=1e-8)
    assert e.value.code == 6
    s.set_wait_polls(0)
    again = s.solve(b, tol=1e-8)
    assert torch.equal(again[0], x) and again[1:3] == (iters, status)


@pytest.mark.parametrize("precision", ["fp32", "fp32_bf16"])
def test_chunk_heights_are_timed_on_the_sweeps_that_run(precision):
    """Autotuned layouts in FP32 modes, level 1 swept by colour launches and the others by flow: sound, and a
    solve in as many iterations as with the rule's heights, to one (the rounding of the sums differs)."""
    p = inputs.small_3d(128, 128, 64, seed=99)
    b = torch.tensor(inputs.random_vector(p.n, 100), device=DEV)
    s, t = (solver(p, precision=precision, ic_order="colour", autotune=a) for a in (True, False))
    c = s.check_layouts()
    assert c.pop("layouts") == 3 * (s.nlevels - 1) + 3 and not any(c.values())
    x, iters, status, _ = s.solve(b, tol=1e-8)
    _, rule, _, _ = t.solve(b, tol=1e-8)
    assert status == 0 and abs(iters - rule) <= 1
    assert float((b - s.spmv(x)).norm() / b.norm()) <= 2e-8


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_one_handle_takes_batched_calls_of_every_kind(precision):
    """The batched graph is kept by padded width and kind and replayed: on one handle, calls of other
    right-hand sides, widths within one padding and across paddings, tolerances, limits and kinds give what
    a fresh handle gives, to the bit."""
    p = inputs.small_3d(19, 17, 9, seed=97)
    make = lambda: solver(p, coarse_max=64, ic_order="colour", precision=precision)      # noqa: E731

    def call(s, kind, K, tol, maxit):
        B = torch.tensor(np.ascontiguousarray(inputs.batch_rhs(p.n, K, cells_per_rhs=4, seed=98 + K).T), device=DEV)
        if kind == "block":
            X, it, _, st = s.solve_block(B, tol=tol, maxit=maxit)
            return [X], [it, st]
        if kind == "adjoint":
            X, L, itf, ita = s.solve_batched_adjoint(B, tol=tol, maxit=maxit)
            return [X, L], [itf.tolist(), ita.tolist()]
        X, it, st = s.solve_batched(B, tol=tol, maxit=maxit)
        return [X], [it.tolist(), st.tolist()]

    s = make()
    for args in [("batched", 16, 1e-6, 100), ("batched", 9, 1e-8, 100), ("adjoint", 9, 1e-6, 100), ("block", 12, 1e-6, 100),
                 ("batched", 16, 1e-8, 3), ("batched", 12, 1e-8, 100), ("adjoint", 40, 1e-8, 100), ("adjoint", 33, 1e-6, 100),
                 ("block", 33, 1e-6, 100), ("batched", 5, 1e-6, 100), ("batched", 16, 1e-6, 100)]:
        fresh = make()
        (tensors, numbers), (want, count) = call(s, *args), call(fresh, *args)
        assert numbers == count, args
        assert all(torch.equal(a, b) for a, b in zip(tensors, want)), args
        fresh.close()


def test_chunk_heights_do_not_depend_on_the_precision():
    """The rule for the chunk height of a widest colour that takes two waves of blocks goes by the FP64 kernel's
    occupancy: 8 entries to a lane leave 9 blocks of four chunks on an SM.  FP32 modes take the same heights, so
    that every sum keeps its order (a colour of many waves, in FP64 alone, is left out by the sizes)."""
    sms = torch.cuda.get_device_properties(DEV).multi_processor_count
    for shape in [(61, 53, 37), (112, 112, 56), (128, 128, 64)]:
        p = inputs.small_3d(*shape, seed=101)
        hs = [solver(p, precision=q) for q in ("fp64", "fp32", "fp32_bf16")]
        for l in range(1, hs[0].nlevels - 1):
            if hs[0].level_info(l)["n"] // hs[0].level_info(l)["ncolours"] < 4 * 8 * 4 * sms:
                assert len({s.level_layout(l)["C"] for s in hs}) == 1, (shape, l)


def test_two_colours_without_diagonals():
    """A grid in a random order: two colours, no diagonal form, so whole rows of P and R.  The same as the
    oracle's application up to the rounding of the sums (a relative 1e-11, as for the other layouts)."""
    import oracle as O
    A = O.tpfa_problem(inputs.small_3d(40, 36, 1, seed=102))
    n = A.rowptr.size - 1
    new = np.random.default_rng(103).permutation(n)
    rows = new[np.repeat(np.arange(n), np.diff(A.rowptr))]
    o = np.lexsort((new[A.col], rows))
    ptr = np.concatenate(([0], np.cumsum(np.bincount(rows, minlength=n)))).astype(np.int32)
    csr = ptr, new[A.col][o].astype(np.int32), A.val[o]
    orc = O.Oracle(O.Csr(n, *csr), coarse_max=64)
    s = cpc.Solver(*csr, coarse_max=64)
    assert s.level_info(0)["ncolours"] == 2 and s.level_layout(0)["ndiag"] == 0
    r = inputs.random_vector(n, 104)
    for which, op in (("bco", O.BCO), ("amg", O.STILDE)):
        z, ref = s.apply(torch.tensor(r, device=DEV), which).cpu().numpy(), orc.apply(op, r)
        assert np.linalg.norm(z - ref) / np.linalg.norm(ref) < 1e-11
    B = torch.tensor(np.stack((r, 2.0 * r), 1), device=DEV)
    X, it, st = s.solve_batched(B, tol=1e-10)
    x, iters, _, _ = s.solve(B[:, 0].contiguous(), tol=1e-10)
    assert not st.any() and it[0] == it[1] == iters and float((X[:, 0] - x).norm() / x.norm()) <= 1e-11
