"""The greedy colouring at the edges of its kernel: equal to the oracle's, colour for colour.

A block takes four points and a warp one, 32 entries of its row at a time and 64 colours at a time.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle as O  # noqa: E402
from paper_1205_6113_gb300 import cpc  # noqa: E402

pytestmark = pytest.mark.gpu


def cliques(sizes, seed):
    """Disjoint complete graphs of the given sizes in a random order, a chain through their first points."""
    n = int(np.sum(sizes))
    name = np.random.default_rng(seed).permutation(n)
    D = np.zeros((n, n))
    first = np.cumsum(sizes) - sizes
    for f, m in zip(first, sizes):
        q = name[f:f + m]
        D[np.ix_(q, q)] = -1.0
    D[name[first[1:]], name[first[:-1]]] = D[name[first[:-1]], name[first[1:]]] = -0.5
    np.fill_diagonal(D, 0.0)
    np.fill_diagonal(D, 0.5 - D.sum(1))
    r, c = np.nonzero(D)
    ptr = np.concatenate(([0], np.cumsum(np.bincount(r, minlength=n))))
    return n, ptr.astype(np.int32), c.astype(np.int32), D[r, c]


@pytest.mark.parametrize("sizes", [[3], [3, 1], [4, 3, 2], [32, 1], [33, 2], [34, 31], [64, 1], [65, 3], [66, 129, 2]])
def test_greedy_colours_match_the_oracle(sizes):
    n, ptr, col, val = cliques(np.array(sizes), seed=sum(sizes))
    s = cpc.Solver(ptr, col, val, coarse_max=1)
    orc = O.Oracle(O.Csr(n, ptr, col, val), coarse_max=1)
    _, colour = s.level_splitting(0)
    assert np.array_equal(colour, orc.level_cf_colour(0)[1])
    assert colour.max() + 1 == max(sizes)


def test_greedy_colours_a_long_chain_of_long_rows():
    """A coarse level whose points are all coupled: each takes its colour after all before it, half a
    second later for the last.  The fine level has a point for each pair of the first m, so that those
    m become the coarse points."""
    m = 2200
    a, b = np.triu_indices(m, 1)
    f = m + np.arange(a.size)
    r, c = np.concatenate((a, b, f, f)), np.concatenate((f, f, a, b))
    n = m + a.size
    r, c = np.concatenate((r, np.arange(n))), np.concatenate((c, np.arange(n)))
    v = np.where(r == c, np.where(r < m, float(m), 2.5), -1.0)
    o = np.lexsort((c, r))
    ptr = np.concatenate(([0], np.cumsum(np.bincount(r, minlength=n)))).astype(np.int32)
    s = cpc.Solver(ptr, c[o].astype(np.int32), v[o], coarse_max=64)
    i = s.level_info(1)
    assert i["n"] == m and i["nnz"] == m * m
    assert np.array_equal(np.sort(s.level_splitting(1)[1]), np.arange(m))


def chain(order):
    """Cells in a row, the k-th one numbered order[k]."""
    n = order.size
    r = np.concatenate((order, order[1:], order[:-1]))
    c = np.concatenate((order, order[:-1], order[1:]))
    v = np.concatenate((np.full(n, 2.5), np.full(2 * n - 2, -1.0)))
    o = np.lexsort((c, r))
    ptr = np.concatenate(([0], np.cumsum(np.bincount(r, minlength=n)))).astype(np.int32)
    return ptr, c[o].astype(np.int32), v[o]


@pytest.mark.parametrize("n", [2, 9, 257, 4097])
@pytest.mark.parametrize("numbering", ["up", "down", "random"])
def test_chain_colours_match_the_oracle(n, numbering):
    order = {"up": np.arange(n), "down": np.arange(n)[::-1], "random": np.random.default_rng(n).permutation(n)}[numbering]
    csr = chain(order)
    s = cpc.Solver(*csr, coarse_max=1)
    orc = O.Oracle(O.Csr(n, *csr), coarse_max=1)
    for l in range(s.nlevels - 1):
        assert np.array_equal(s.level_splitting(l)[1], orc.level_cf_colour(l)[1])


def test_a_long_chain_is_not_walked_link_by_link():
    """200,000 cells in a row: two colours, in far less than the 16-27 ms of joining them one by one (0.2 ms)."""
    n = 200000
    csr = chain(np.arange(n))
    ms = []
    for _ in range(3):
        s = cpc.Solver(*csr)
        ms.append(s.setup_phases_ms()["colouring"])
        colour = s.level_splitting(0)[1]
        s.close()
    assert np.array_equal(colour, np.arange(n) % 2)
    assert min(ms) < 5.0, ms
