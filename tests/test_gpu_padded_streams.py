"""Systems with fields of unequal size, which run padded: setup on one stream,
cycle and solve on others, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2103_07537_gb300 import bamg, problems as P

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("b,fields", [(3, [0, 0, 1]), (4, [0, 0, 0, 1])])
def test_padded_system_on_other_streams_than_its_setup(b, fields):
    s = P.random_block_system(21, b, fields, seed=b)
    kw = dict(max_levels=3, max_coarse=0)
    o = oracle.Hierarchy.from_system(s, **kw)
    r = np.random.default_rng(b).standard_normal(s.n_unknowns)
    d = [dev(a) for a in (s.row_ptr, s.col_idx, s.vals.reshape(-1))]
    rd, bd = dev(r), dev(s.rhs)
    z, x = torch.zeros_like(rd), torch.zeros_like(rd)
    setup, cycle, solve = (torch.cuda.Stream() for _ in range(3))
    torch.cuda.synchronize()
    g = bamg.Solver(*d, b, fields, stream=setup.cuda_stream, **kw)
    g.apply(rd, z, stream=cycle.cuda_stream)
    cycle.synchronize()
    want = o.vcycle(r)
    assert np.abs(z.cpu().numpy() - want).max() <= 1e-12 * np.abs(want).max()
    st, it, rr = g.solve(bd, x, tol=1e-8, restart=30, max_iter=500, stream=solve.cuda_stream)
    assert st == bamg.BAMG_OK and abs(it - o.fgmres(s.rhs, tol=1e-8, restart=30, max_iter=500)[1]) <= 1
