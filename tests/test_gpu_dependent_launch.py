"""Cycles whose kernels start while their predecessors drain against the same
cycles in plain launches: the same kernels in the same order, so the same bits,
for every sub-solver, with and without the graph, from the first cycle on."""
import numpy as np
import pytest

from paper_2103_07537_gb300 import bamg, problems as P

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


VARIANTS = {
    "warp": dict(autotune=0),
    "thread": dict(autotune=2),
    "thread_split": dict(autotune=4),
    "inner_sweeps": dict(autotune=0, inner_sweeps=3),
    "ilu": dict(autotune=0, sub_solver=1),
    "schwarz": dict(autotune=0, sub_solver=2),
    "smoothed_p": dict(autotune=0, smooth_p=1),
}


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("name", list(VARIANTS))
@pytest.mark.parametrize("b,fields", [(3, [0] * 3), (4, [0, 0, 1, 1])])
def test_same_bits_as_plain_launches(b, fields, name, prec):
    s = P.random_block_system(60, b, fields, seed=b)
    rp, ci, va = dev(s.row_ptr), dev(s.col_idx), dev(s.vals.reshape(-1))
    r = dev(np.random.default_rng(1).standard_normal(s.n_unknowns))
    out = []
    for pdl, graph in ((0, 0), (1, 1), (1, 0)):
        g = bamg.Solver(rp, ci, va, s.b, s.field_of_dof, max_levels=4, max_coarse=0, cycle_prec=prec, use_pdl=pdl,
                        use_graph=graph, **VARIANTS[name])
        for _ in range(3):
            z = torch.zeros_like(r)
            g.apply(r, z)
            out.append(z.cpu().numpy())
    assert np.all(np.isfinite(out[0]))
    for z in out[1:]:
        assert np.array_equal(z, out[0])
