"""The coarse levels of a cycle as one cluster launch: the V-cycle against the
oracle over block shapes, sweeps, levels of fewer nodes than the cluster has
CTAs, per-node damping set later, and FP32; repeated cycles bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2103_07537_gb300 import bamg, problems as P

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def solver(s, **kw):
    return bamg.Solver(dev(s.row_ptr), dev(s.col_idx), dev(s.vals.reshape(-1)), s.b, s.field_of_dof, **kw)


def apply(g, r):
    z = torch.empty(r.size, dtype=torch.float64, device="cuda")
    g.apply(dev(r), z)
    torch.cuda.synchronize()
    return z.cpu().numpy()


def rel_max(a, ref):
    return np.abs(a - ref).max() / np.abs(ref).max()


SHAPES = [(1, [0]), (2, [0] * 2), (3, [0] * 3), (4, [0] * 4), (4, [0, 0, 1, 1]), (5, [0] * 5), (6, [0] * 6),
          (6, [0, 0, 0, 1, 1, 1]), (6, [0, 0, 1, 1, 2, 2]), (7, [0] * 7), (8, [0] * 8), (8, [0] * 4 + [1] * 4),
          (8, [0, 0, 1, 1, 2, 2, 3, 3])]


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("b,fields", SHAPES)
def test_every_block_shape(b, fields, prec):
    s = P.random_block_system(17, b, fields, seed=20 + b)  # 289 nodes: uneven slices
    kw = dict(max_levels=4, max_coarse=0)
    g = solver(s, cycle_prec=prec, **kw)
    assert g.stats()["coarse_cycle_level"] >= 0
    r = np.random.default_rng(b).standard_normal(s.n_unknowns)
    z = apply(g, r)
    want = oracle.Hierarchy.from_system(s, **kw).vcycle(r)
    # FP64: the bar of every V-cycle test; FP32: sums of at most 9 b products and
    # 3 levels of them, 2^-24 each, on a diagonally dominant system
    assert rel_max(z, want) <= (1e-12 if prec == 64 else 3 * 9 * b * 2.0 ** -24)
    for _ in range(3):
        assert np.array_equal(apply(g, r), z)


@pytest.mark.parametrize("variant", [dict(n_pre=0, n_post=1), dict(n_pre=1, n_post=0), dict(n_pre=0, n_post=0),
                                     dict(n_pre=2, n_post=3, omega=0.7)])
@pytest.mark.parametrize("name", ["stokes2d_32", "mhd2d_13", "stokes3d_7"])
def test_sweeps_and_levels(name, variant):
    s = {"stokes2d_32": lambda: P.stokes2d(32, 1), "mhd2d_13": lambda: P.mhd2d(13, 2),
         "stokes3d_7": lambda: P.stokes3d(7, 3)}[name]()
    kw = dict(max_levels=10, max_coarse=0, **variant)  # down to a few nodes: CTAs without any
    g = solver(s, **kw)
    assert (g.stats()["coarse_cycle_level"] >= 0) == (sum(variant.get(k, 1) for k in ("n_pre", "n_post")) > 0)
    r = np.random.default_rng(3).standard_normal(s.n_unknowns)
    assert rel_max(apply(g, r), oracle.Hierarchy.from_system(s, **kw).vcycle(r)) <= 1e-12


def test_part_of_the_levels_and_solve():
    s = P.mhd2d(64, 1)
    kw = dict(max_levels=4, max_coarse=0)
    g, o = solver(s, **kw), oracle.Hierarchy.from_system(s, **kw)
    assert g.stats()["coarse_cycle_level"] >= 1
    r = np.random.default_rng(5).standard_normal(s.n_unknowns)
    z = apply(g, r)
    assert rel_max(z, o.vcycle(r)) <= 1e-12
    assert np.array_equal(z, apply(solver(s, use_graph=0, **kw), r))
    x = torch.zeros(s.n_unknowns, dtype=torch.float64, device="cuda")
    st, it, rr = g.solve(dev(s.rhs), x, tol=1e-8, restart=30, max_iter=2000)
    assert st == bamg.BAMG_OK and abs(it - o.fgmres(s.rhs, tol=1e-8, restart=30, max_iter=2000)[1]) <= 1


def test_large_coarsest_system_keeps_its_launches():
    s = P.stokes2d(65, 1)  # 484 coarsest nodes: a product of 1452 rows
    g = solver(s, max_levels=10, max_coarse=2500, cycle_prec=32, coarse_prec=32)
    assert g.stats()["coarse_cycle_level"] == -1


def test_damping_replaced_after_setup():
    s = P.mhd2d(24, 3)
    kw = dict(max_levels=3, max_coarse=0)
    g = solver(s, **kw)
    n = [g.level(l)["n"] for l in range(2)]
    w = [np.random.default_rng(l).uniform(0.3, 0.9, (n[l], 2)) for l in range(2)]
    r = np.random.default_rng(9).standard_normal(s.n_unknowns)
    apply(g, r)
    for l in range(2):
        g.set_omega(l, dev(w[l].reshape(-1)))
    torch.cuda.synchronize()
    o = oracle.Hierarchy.from_system(s, omega_s_arr=np.concatenate([a.reshape(-1) for a in w]), **kw)
    assert rel_max(apply(g, r), o.vcycle(r)) <= 1e-12
