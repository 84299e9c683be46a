"""A recorded tuning is taken again for a level of the same shape only, and the
length of the longest row belongs to the shape: a mapping that stages whole
rows in shared memory takes rows up to a length."""
import numpy as np
import pytest

import oracle
from paper_2103_07537_gb300 import bamg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

N = 1234  # nodes: even ones of colour 0, odd ones of colour 1 in both graphs


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def graph(pairs, b):
    """Symmetric block pattern with its diagonal, weakly coupled identity-like blocks."""
    e = np.array(sorted({(i, j) for a, c in pairs for i, j in ((a, c), (c, a))} | {(i, i) for i in range(N)}))
    rp = np.zeros(N + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(e[:, 0], minlength=N))
    ci = e[:, 1].astype(np.int32)
    vals = np.random.default_rng(7).uniform(-1, 1, (ci.size, b, b)) / (2.0 * b)
    diag = e[:, 0] == e[:, 1]
    vals[diag] += (1.0 + np.diff(rp)[e[diag, 0], None, None]) * np.eye(b)
    return rp, ci, vals


def path(b):
    return graph([(i, i + 1) for i in range(N - 1)], b)


def hub(b):
    """As many nodes, blocks and nodes per colour as the path, one row of N / 2 + 1 blocks."""
    return graph([(i - 1, i) for i in range(1, N, 2)] + [(0, i) for i in range(3, N, 2)], b)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("b", [1, 3, 6])
def test_longest_row_is_part_of_the_shape(b, prec):
    g1, g2 = path(b), hub(b)
    assert g1[1].size == g2[1].size and np.diff(g2[0]).max() == N // 2 + 1
    for g in (g1, g2):
        assert np.array_equal(oracle.colour(g[0], g[1])[0], np.arange(N) % 2)
    kw = dict(max_levels=2, max_coarse=0)

    def solver(g):
        return bamg.Solver(dev(g[0]), dev(g[1]), dev(g[2].reshape(-1)), b, [0] * b, cycle_prec=prec, **kw)

    first, other, again = solver(g1), solver(g2), solver(g2)
    cached = [s.stats()["levels"][0]["tune_cached"] for s in (first, other, again)]
    assert cached == [0, 0, 1]
    assert again.stats()["levels"][0]["smoother_mapping"] == other.stats()["levels"][0]["smoother_mapping"]
    r = dev(np.random.default_rng(b).standard_normal(N * b))
    z = [torch.zeros_like(r) for _ in range(2)]
    for s, out in zip((other, again), z):
        s.apply(r, out)
    assert torch.isfinite(z[0]).all() and torch.equal(z[0], z[1])
