"""A forced sweep builds its plan once: a hierarchy whose tuning is on record
holds as much device memory as the one that was tuned."""
import numpy as np
import pytest

from paper_2103_07537_gb300 import bamg, problems as P

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("sweep", [2, 3])
@pytest.mark.parametrize("b,fields", [(3, [0] * 3), (4, [0, 0, 1, 1])])
def test_recorded_tuning_takes_the_same_memory(b, fields, sweep):
    s = P.random_block_system(47, b, fields, seed=11)
    rp, ci, va = dev(s.row_ptr), dev(s.col_idx), dev(s.vals.reshape(-1))
    runs = [bamg.Solver(rp, ci, va, s.b, s.field_of_dof, max_levels=3, max_coarse=0, sweep=sweep) for _ in range(2)]
    st = [g.stats() for g in runs]
    assert [l["tune_cached"] for l in st[1]["levels"][:-1]] == [1, 1]
    assert all(l["smoother_mapping"].startswith("sweep") for q in st for l in q["levels"][:-1])
    assert st[1]["device_bytes"] <= st[0]["device_bytes"]
    r = dev(np.random.default_rng(2).standard_normal(s.n_unknowns))
    z = [torch.zeros_like(r) for _ in range(2)]
    for g, out in zip(runs, z):
        g.apply(r, out)
    assert torch.equal(z[0], z[1])
