"""What the first setup of a level shape pays for its tuning: each mapping once
alone and once as the cycle runs it, in a bounded number of launches."""
import numpy as np
import pytest

from paper_2103_07537_gb300 import bamg, problems as P

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("n_side,b", [(35, 3), (46, 4), (61, 2)])
def test_launches_of_a_tuned_setup(n_side, b, prec):
    s = P.random_block_system(n_side, b, [0] * b, seed=2)
    d = [dev(a) for a in (s.row_ptr, s.col_idx, s.vals.reshape(-1))]
    counts = []
    for _ in range(2):
        before = bamg.amg_launch_count()
        g = bamg.Solver(*d, b, s.field_of_dof, max_levels=4, max_coarse=0, cycle_prec=prec)
        counts.append(bamg.amg_launch_count() - before)
        st = g.stats()
        del g
    levels = st["levels"][:-1]
    assert [l["tune_cached"] for l in levels] == [1] * len(levels)
    # a candidate: one launch, three and ten (five for whole steps) more.  Alone: 8 mappings of the smoother and 2
    # of the residual; as the cycle runs them: 4 mappings, a step from zero and one from an iterate; the chosen
    # mapping against two sweeps; 3 of the outer product, once; 10 a level for the sweep's plan and its tiles
    most = sum(14 * 10 + 9 * 4 * 2 * l["colours"] + 14 * (l["colours"] + 2) + 10 for l in levels) + 14 * 3
    assert counts[0] - counts[1] <= most
