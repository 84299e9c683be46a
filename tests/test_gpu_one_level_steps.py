"""Solves of one level, whose cycle is the coarsest solve, project twice in every
step, and say so before the first outcome is read: the step's launches are those
of two projections that are always taken, plus the second one's own product."""
import numpy as np
import pytest

import oracle
from paper_2103_07537_gb300 import bamg, problems as P

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("name", ["stokes2d", "mhd2d", "stokes3d"])
def test_launches_of_a_one_level_solve(name):
    s = {"stokes2d": lambda: P.stokes2d(16, 1), "mhd2d": lambda: P.mhd2d(12, 1), "stokes3d": lambda: P.stokes3d(6, 1)}[name]()
    launches = []
    for ortho in (0, 1):  # a second projection where it is due, always
        g = bamg.Solver(dev(s.row_ptr), dev(s.col_idx), dev(s.vals.reshape(-1)), s.b, s.field_of_dof, ortho=ortho)
        assert g.num_levels == 1
        x = torch.zeros(s.n_unknowns, dtype=torch.float64, device="cuda")
        g.solve(dev(s.rhs), x, tol=1e-8, restart=30, max_iter=100)  # (the cycle's graph is captured here)
        x.zero_()
        before = bamg.amg_launch_count()
        st, it, rr = g.solve(dev(s.rhs), x, tol=1e-8, restart=30, max_iter=100)
        launches.append(bamg.amg_launch_count() - before)
        q = g.stats()
        assert st == bamg.BAMG_OK and rr <= 1e-8 and it == 1
        assert q["second_projections"] == q["arnoldi_steps"] == 1
        assert abs(it - oracle.Hierarchy.from_system(s).fgmres(s.rhs, tol=1e-8, restart=30, max_iter=100)[1]) <= 1
    assert launches[0] - launches[1] == 1


def test_no_cycle_ahead_of_an_outcome_that_ends_the_solve():
    """Two FP32 solves of two steps, whose first steps reduce the residual by different amounts: a
    cycle started ahead of the second one's outcome would show as launches of one of them only."""
    launches = []
    for n in (16, 24):
        s = P.stokes2d(n, 1)
        g = bamg.Solver(dev(s.row_ptr), dev(s.col_idx), dev(s.vals.reshape(-1)), s.b, s.field_of_dof, cycle_prec=32)
        assert g.num_levels == 1
        x = torch.zeros(s.n_unknowns, dtype=torch.float64, device="cuda")
        g.solve(dev(s.rhs), x, tol=1e-8, restart=30, max_iter=100)
        x.zero_()
        before = bamg.amg_launch_count()
        st, it, rr = g.solve(dev(s.rhs), x, tol=1e-8, restart=30, max_iter=100)
        launches.append(bamg.amg_launch_count() - before)
        assert st == bamg.BAMG_OK and rr <= 1e-8 and it == 2
    assert launches[0] == launches[1]
