"""The colouring of a level is one launch whatever the level's size: setups on
either side of the size up to which 255 colours are allowed count alike."""
import numpy as np
import pytest

import oracle
from paper_2103_07537_gb300 import bamg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def path(n):
    row = np.repeat(np.arange(n), 3)
    col = row + np.tile([-1, 0, 1], n)
    keep = (col >= 0) & (col < n)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(row[keep], minlength=n))
    return rp, col[keep].astype(np.int32), np.where(row == col, 4.0, -1.0)[keep]


def test_launches_do_not_depend_on_the_colour_limit():
    counts = []
    for n in (39999, 40001):
        rp, ci, va = path(n)
        d = [dev(a) for a in (rp, ci, va)]
        before = bamg.amg_launch_count()
        g = bamg.Solver(*d, 1, [0], max_levels=12, autotune=0)
        counts.append((bamg.amg_launch_count() - before, g.num_levels))
        assert np.array_equal(g.level(0)["colour"], oracle.colour(rp, ci)[0])
    assert counts[0] == counts[1]
