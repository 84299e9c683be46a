"""Aggregation and colouring of graphs that sit at the edges of their chunks of
256 nodes, or make their dependency chains as long or as dense as they can be,
against the oracle's sequential rules, bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2103_07537_gb300 import bamg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def csr(n, pairs):
    """Structurally symmetric pattern with its diagonal from (i, j) pairs."""
    e = np.array(sorted({(int(a), int(b)) for i, j in pairs for a, b in ((i, j), (j, i))} | {(i, i) for i in range(n)}))
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(e[:, 0], minlength=n))
    return rp, e[:, 1].astype(np.int32)


def path(n, order=None):
    p = np.arange(n) if order is None else order
    return csr(n, zip(p[:-1], p[1:]))


def random_graph(n, m, seed):
    r = np.random.default_rng(seed)
    return csr(n, r.integers(0, n, (m, 2)))


GRAPHS = {
    "path_255": lambda: path(255),
    "path_256": lambda: path(256),
    "path_257": lambda: path(257),
    "path_5000": lambda: path(5000),  # every node waits for the one before it
    "path_backward": lambda: path(1000, np.arange(1000)[::-1]),
    "path_permuted": lambda: path(3000, np.random.default_rng(1).permutation(3000)),
    "clique_100": lambda: csr(100, [(i, j) for i in range(100) for j in range(i)]),  # 100 colours
    "star": lambda: csr(700, [(699, j) for j in range(699)]),  # one row of 700 blocks
    "random_sparse": lambda: random_graph(4097, 6000, 2),
    "random_dense": lambda: random_graph(1500, 30000, 3),
}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_graph_rules_match_sequential_oracle(name):
    rp, ci = GRAPHS[name]()
    n = rp.size - 1
    row = np.repeat(np.arange(n), np.diff(rp))
    vals = np.where(row == ci, 4.0 + np.diff(rp)[row], -1.0)
    g = bamg.Solver(dev(rp), dev(ci), dev(vals), 1, [0], max_levels=2, max_coarse=0, autotune=0)
    want_agg, _, want_n = oracle.aggregate(rp, ci)
    L = g.level(0)
    assert np.array_equal(L["agg"], want_agg) and L["n_agg"] == want_n
    assert np.array_equal(L["colour"], oracle.colour(rp, ci)[0])
