"""amg_stats counts the launches that decided a level's aggregates and colours:
one each on every level with a smoother, none on the coarsest."""
import numpy as np
import pytest

from paper_2103_07537_gb300 import bamg, problems as P

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def test_rounds_of_every_level():
    s = P.random_block_system(30, 3, [0] * 3, seed=1)
    g = bamg.Solver(dev(s.row_ptr), dev(s.col_idx), dev(s.vals.reshape(-1)), s.b, s.field_of_dof, max_levels=3,
                    max_coarse=0, autotune=0)
    levels = g.stats()["levels"]
    assert len(levels) == 3
    for key in ("aggregation_rounds", "colouring_rounds"):
        assert [l[key] for l in levels] == [1, 1, 0]
