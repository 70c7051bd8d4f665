"""The FP32 and BF16 sweeps that run as one launch ordered by their data, against the cycle in 64 bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_1205_6113_gb300 import cpc, inputs  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def neighbour_matrix(pairs, n, seed):
    """SPD CSR with random couplings in [-1.5, -0.5] on the given pairs and a diagonal of 1.5 times their sum."""
    import scipy.sparse as sp
    a, b = pairs
    w = -np.random.default_rng(seed).uniform(0.5, 1.5, a.size)
    A = sp.coo_matrix((np.tile(w, 2), (np.concatenate((a, b)), np.concatenate((b, a)))), shape=(n, n)).tocsr()
    A = A + sp.diags(-1.5 * np.asarray(A.sum(1)).ravel())
    A = A.tocsr()
    A.sort_indices()
    return A


def box_pairs(nx, ny, nz, r):
    i = np.arange(nx * ny * nz)
    x, y, z = i % nx, i // nx % ny, i // (nx * ny)
    a, b = [], []
    for dz in range(-min(r, nz - 1), min(r, nz - 1) + 1):
        for dy in range(-r, r + 1):
            for dx in range(-r, r + 1):
                j = i + dx + nx * (dy + ny * dz)
                ok = (x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) & (z + dz >= 0) & (z + dz < nz) & (j > i)
                a.append(i[ok])
                b.append(j[ok])
    return np.concatenate(a), np.concatenate(b)


def random_pairs(n, m, seed):
    rng = np.random.default_rng(seed)
    p = np.unique(np.sort(rng.integers(0, n, (n * m // 2, 2)), axis=1), axis=0)
    p = p[p[:, 0] != p[:, 1]]
    return p[:, 0], p[:, 1]


def two_cycles(levels, ainv, r, mistake=None):
    """The two V-cycles of "amg" in 64 bits.  levels: (A, P, colour) with the stored values.  mistake: what a
    sweep of the second cycle would do wrong, "zero": old values taken as zero, "mixed": the backward sweep's
    old values taken from its own output before it is written."""
    def sweep(A, colour, f, old, order, forget=False):
        x = old.copy()
        D = A.diagonal()
        done = np.zeros(A.shape[0], dtype=bool)
        for c in order:
            rows = np.flatnonzero(colour == c)
            src = np.where(done, x, 0.0) if forget else x
            x[rows] = (f[rows] - (A[rows] @ src - D[rows] * src[rows])) / D[rows]
            done[rows] = True
        return x

    def cycle(l, f, x, wrong):
        if l == len(levels):
            return ainv @ f
        A, P, colour = levels[l]
        g = colour.max() + 1
        x = sweep(A, colour, f, x, range(g), wrong == "zero" and l == 0)
        x = x + P @ cycle(l + 1, P.T @ (f - A @ x), np.zeros(P.shape[1]), wrong)
        return sweep(A, colour, f, x, range(g - 1, -1, -1), wrong == "mixed" and l == 0)

    z = cycle(0, r, np.zeros_like(r), None)
    return cycle(0, r, z, mistake)


@pytest.mark.parametrize("precision", ["fp32", "fp32_bf16"])
@pytest.mark.parametrize("name", ["9 points", "27 points", "125 points", "220 random"])
def test_fp32_sweeps_match_the_cycle_in_64_bits(name, precision):
    """FP32 sweeps by flow, whose rows hold new and old values mixed: forward from zero, forward from a given
    iterate and backward, with 4 to 28 entries to a lane, against the same two cycles in 64 bits on the
    stored values.  A row's sum of k terms to a lane is off by at most e = (k + 8) u of its magnitudes, u = 2^-24
    (k products, the lanes' tree, the update).  Rows are 1.5 times dominant, so a sweep adds at most 5 e max |x|,
    and the coarse correction, a projection applied to a residual off by as much, about 10 e: 20 e for the
    two sweeps and the correction of a level, over three levels and two cycles 120 e, and 150 e is asked.  A
    sweep that takes a wrong old value is off by more than three times that, which is checked in 64 bits."""
    import scipy.sparse as sp
    n, pairs = {"9 points": (1440, lambda: box_pairs(40, 36, 1, 1)), "27 points": (1320, lambda: box_pairs(12, 11, 10, 1)),
                "125 points": (1080, lambda: box_pairs(12, 10, 9, 2)), "220 random": (900, lambda: random_pairs(900, 220, 94))}[name]
    A = neighbour_matrix(pairs(), n, 95)
    s = cpc.Solver(A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, precond="amg", precision=precision, coarse_max=64)
    f32 = lambda M: sp.csr_matrix((M[2].astype(np.float32).astype(np.float64), M[1], M[0]), shape=M[3])   # noqa: E731
    levels, k = [], 0
    for l in range(s.nlevels):
        ptr, col, val = s.level_matrix(l)
        nl = ptr.size - 1
        if l == s.nlevels - 1:
            ainv = np.linalg.inv(sp.csr_matrix((val, col, ptr), shape=(nl, nl)).toarray())
            break
        S = f32((ptr, col, val, (nl, nl)))
        if l and precision == "fp32_bf16":
            rows = np.repeat(np.arange(nl), np.diff(ptr))
            b = torch.tensor(val, dtype=torch.float64).to(torch.bfloat16).double().numpy()
            S = sp.csr_matrix((np.where(rows == col, S.data, b), col, ptr), shape=(nl, nl))
        pp, pc, pv = s.level_interp(l)
        levels.append((S, f32((pp, pc, pv, (nl, s.level_info(l)["nc"]))), s.level_splitting(l)[1]))
        k = max(k, -(-int(np.diff(ptr).max()) * s.level_layout(l)["C"] // 32))
    r = inputs.random_vector(n, 96)
    ref = two_cycles(levels, ainv, r)
    bound = 150 * (k + 8) * 2.0 ** -24 * np.abs(ref).max()
    for mistake in ("zero", "mixed"):
        assert np.abs(two_cycles(levels, ainv, r, mistake) - ref).max() > 3 * bound
    z = s.apply(torch.tensor(r, device=DEV)).cpu().numpy()
    assert np.abs(z - ref).max() <= bound
