"""Aggregation and colouring of graphs with more nodes than the launch has in
work at once (608 chunks of 256 on 152 SMs), so that every CTA takes further
chunks and waits reach across the whole window, against the oracle's sequential
rules, bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2103_07537_gb300 import bamg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def band(n, width, order):
    """Node order[i] coupled with order[i + 1], ..., order[i + width]; symmetric, with its diagonal."""
    i = np.concatenate([order] + [order[:-w] for w in range(1, width + 1)] + [order[w:] for w in range(1, width + 1)])
    j = np.concatenate([order] + [order[w:] for w in range(1, width + 1)] + [order[:-w] for w in range(1, width + 1)])
    k = np.lexsort((j, i))
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(i, minlength=n))
    return rp, j[k].astype(np.int32)


def local_permutation(n, window, seed):
    r = np.random.default_rng(seed)
    return np.concatenate([a + r.permutation(min(window, n - a)) for a in range(0, n, window)])


GRAPHS = {
    # one chain through all nodes, ascending; and the same chain walked downwards
    "path": lambda: band(200001, 1, np.arange(200001)),
    "path_backward": lambda: band(160000, 1, np.arange(160000)[::-1]),
    # waits into earlier chunks, of a few chunks' and of half a window's reach
    "band_permuted_near": lambda: band(170003, 3, local_permutation(170003, 1000, 1)),
    "band_permuted_far": lambda: band(311296, 2, local_permutation(311296, 80000, 2)),
}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_long_chains_match_sequential_oracle(name):
    rp, ci = GRAPHS[name]()
    n = rp.size - 1
    assert n > 608 * 256
    row = np.repeat(np.arange(n), np.diff(rp))
    vals = np.where(row == ci, 4.0 + np.diff(rp)[row], -1.0)
    g = bamg.Solver(dev(rp), dev(ci), dev(vals), 1, [0], max_levels=12, autotune=0)
    want_agg, _, want_n = oracle.aggregate(rp, ci)
    L = g.level(0)
    assert np.array_equal(L["agg"], want_agg) and L["n_agg"] == want_n
    assert np.array_equal(L["colour"], oracle.colour(rp, ci)[0])
    phase = g.stats()["setup_phase_ms"]
    print(name, {k: round(v, 2) for k, v in phase.items()})
