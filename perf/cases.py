"""What a user of this framework has it do, as cases that can be timed and compared.

A case is one call (or one short sequence of calls) through the public entry
points of ``paper_2103_07537_gb300.bamg`` on a system of the kinds that the
repository's benchmark and tests use: Stokes-type systems in 2D and 3D, the
coupled four-field system in 2D (with one resistivity or one per cell), mixed
Q2/Q1 elements, and batches.

* ``cycle``: one V-cycle on a hierarchy that the program keeps: the step that a
  Krylov method of the program's own repeats.  An FP32 cycle computes FP32
  numbers and widens them on exit; a program that keeps its correction in FP32
  takes them back, which loses nothing, and that is what comes back here.
* ``setup``: a new matrix: hierarchy, first cycle, release, as once per Newton
  or time step.
* ``solve``: FGMRES to a relative residual of 1e-8 from a zero guess.
* ``host``: the whole call on host buffers (copies, setup, solve, copy back).
* ``spmv``: the block-CSR product on its own.
* ``train``: one step of the damping network's training (gradient and Adam).

The matrices are assembled on the GPU from the seed (random right-hand sides,
viscosities, resistivities and background fields); ``exact`` has a V-cycle of
its own in plain torch, in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2103_07537_gb300 import bamg, learn, problems

TOL, MAX_ITER = 1e-8, 400


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest configuration of the repository: latency and launches
        dict(name="cycle_stokes2d_32", kind="cycle", system="stokes2d", N=32, prec=64, levels=3, max_coarse=0),
        # the 2D four-field configuration in the default FP64 cycle
        dict(name="cycle_mhd2d_128", kind="cycle", system="mhd2d", N=128, prec=64, levels=4, max_coarse=0),
        # the benchmark's default workload: 1.1 M unknowns, the FP32 cycle
        dict(name="cycle_stokes3d_64", kind="cycle", system="stokes3d", N=64, prec=32, levels=10, max_coarse=2500),
        # many independent systems of uneven sizes in one FP32 cycle
        dict(name="cycle_batch48", kind="cycle", system="batch", nsys=48, lo=16, hi=160, prec=32, levels=4,
             max_coarse=0),
        # learned damping and smoothed transfers on the system with a resistivity per cell
        dict(name="cycle_learned_256", kind="cycle", system="cells", N=256, prec=32, levels=10, max_coarse=2500),
        # mixed elements with the paper's own sub-solver (restricted Schwarz)
        dict(name="cycle_q2q1_schwarz_64", kind="cycle", system="q2q1", N=64, prec=32, levels=4, max_coarse=0),
        # a new matrix of the benchmark's default workload
        dict(name="setup_stokes3d_64", kind="setup", system="stokes3d", N=64, prec=32, levels=10, max_coarse=2500),
        # a new matrix of the 2D four-field configuration, FP64
        dict(name="setup_mhd2d_128", kind="setup", system="mhd2d", N=128, prec=64, levels=4, max_coarse=0),
        # the benchmark's default workload solved: FP32 cycle inside FP64 FGMRES(50)
        dict(name="solve_stokes3d_64", kind="solve", system="stokes3d", N=64, prec=32, levels=10, max_coarse=2500,
             restart=50),
        # a ragged 2D size end to end from host buffers, FP64, FGMRES(30)
        dict(name="host_mhd2d_75", kind="host", system="mhd2d", N=75, prec=64, levels=10, max_coarse=2500,
             restart=30),
        # the block-CSR product of the large 3D matrix
        dict(name="spmv_stokes3d_64", kind="spmv", system="stokes3d", N=64),
        # one step of training the damping network, the training program's batch
        dict(name="train_4096", kind="train", rows=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cycle", "cycle", "cycle", "setup", "solve", "host", "spmv", "train"])
    if kind == "train":
        return dict(kind="train", rows=_log_int(rng, 256, 65536))
    system = rng.choice(["stokes2d", "mhd2d", "stokes3d"] if kind != "cycle" else
                        ["stokes2d", "mhd2d", "stokes3d", "stokes3d", "batch", "cells", "q2q1"])
    c = dict(kind=kind, system=system)
    if system == "batch":
        c.update(nsys=_log_int(rng, 2, 48), lo=rng.randint(8, 24), hi=rng.randint(48, 160))
    else:
        lo, hi = {"stokes2d": (16, 256), "mhd2d": (12, 192), "stokes3d": (6, 64), "cells": (64, 256),
                  "q2q1": (12, 64)}[system]
        if kind in ("solve", "host"):
            hi = {"stokes2d": 96, "mhd2d": 96, "stokes3d": 40}[system]
        c["N"] = _log_int(rng, lo, hi)
    if kind == "spmv":
        return c
    c["prec"] = 32 if system in ("cells", "q2q1") else rng.choice([32, 64])
    if kind == "host":
        c["prec"] = 64
    # few levels with a small coarsest solve, or the default coarsening
    c.update(levels=10, max_coarse=2500) if system in ("stokes3d", "cells") or rng.random() < 0.5 else \
        c.update(levels=4, max_coarse=0)
    if kind in ("solve", "host"):
        c["restart"] = rng.choice([30, 50])
    return c


# ---------------------------------------------------------------------------
# inputs: Q1 systems on uniform grids, assembled on the GPU
# ---------------------------------------------------------------------------
def _reference_element(d):
    """Shape values phi[q, l] and gradients dphi[q, l, a] of the d-linear element at its 2^d Gauss points."""
    g = 1.0 / math.sqrt(3.0)
    nl = 2 ** d
    pts = np.array([[g if (q >> a) & 1 else -g for a in range(d)] for q in range(nl)])
    sgn = np.array([[1.0 if (l >> a) & 1 else -1.0 for a in range(d)] for l in range(nl)])
    one = (1.0 + sgn[None] * pts[:, None]) / 2.0  # [q, l, a]
    phi = one.prod(axis=2)
    dphi = np.stack([np.where(np.arange(d) == a, sgn[None] / 2.0, one).prod(axis=2) for a in range(d)], axis=2)
    return phi, dphi, pts


class _Grid:
    """Block pattern of the full node stencil on (N + 1)^d nodes, x fastest, columns ascending."""

    def __init__(self, d, N, dev):
        self.d, self.N, self.m = d, N, N + 1
        n = self.n = self.m ** d
        ids = torch.arange(n, device=dev)
        self.coord = [(ids // self.m ** a) % self.m for a in range(d)]
        off = torch.cartesian_prod(*[torch.tensor([-1, 0, 1], device=dev)] * d).reshape(-1, d).flip(1)
        valid = torch.ones((n, 3 ** d), dtype=torch.bool, device=dev)
        nbr = torch.zeros((n, 3 ** d), dtype=torch.int64, device=dev)
        for a in range(d):
            c = self.coord[a][:, None] + off[None, :, a]
            valid &= (c >= 0) & (c < self.m)
            nbr += c * self.m ** a
        cnt = valid.sum(1)
        self.rp = torch.zeros(n + 1, dtype=torch.int64, device=dev)
        self.rp[1:] = cnt.cumsum(0)
        self.ci = nbr[valid]
        self.row = torch.repeat_interleave(ids, cnt)
        self.pos = self.rp[:-1, None] + valid.cumsum(1) - 1
        self.centre = (3 ** d - 1) // 2
        cells = torch.arange(N ** d, device=dev)
        self.cell = [(cells // N ** a) % N for a in range(d)]
        self.boundary = torch.zeros(n, dtype=torch.bool, device=dev)
        for a in range(d):
            self.boundary |= (self.coord[a] == 0) | (self.coord[a] == N)

    def corner(self, l):
        """Node of local corner l of every cell."""
        return sum((self.cell[a] + ((l >> a) & 1)) * self.m ** a for a in range(self.d))

    def assemble(self, b, block, fixed):
        """Values [nnzb, b, b] from block(la, lc); rows and columns of the fixed dofs [n, b] become identity."""
        vals = torch.zeros((self.ci.numel(), b, b), dtype=torch.float64, device=self.ci.device)
        for la in range(2 ** self.d):
            rows = self.corner(la)
            for lc in range(2 ** self.d):
                code = sum((((lc >> a) & 1) - ((la >> a) & 1) + 1) * 3 ** a for a in range(self.d))
                # every cell of one local pair adds to a block of its own
                k = self.pos[rows, code]
                vals[k] = vals[k] + block(la, lc)
        vals *= (~fixed[self.row])[:, :, None]
        vals *= (~fixed[self.ci])[:, None, :]
        i, r = fixed.nonzero(as_tuple=True)
        vals[self.pos[i, self.centre], r, r] = 1.0
        return vals


def _uniform(gen, *shape):
    return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=gen)


def _stokes(d, N, gen):
    """Q1-Q1 Stokes with pressure stabilisation, viscosity log-uniform in [0.1, 1]."""
    nu = 10.0 ** float(-_uniform(gen, 1))
    g, b, h = _Grid(d, N, "cuda"), d + 1, 1.0 / N
    phi, dphi, _ = _reference_element(d)
    grad, jac = dphi * (2.0 / h), (h / 2.0) ** d
    K = np.einsum("qla,qma->lm", grad, grad) * jac
    G = -np.einsum("qla,qm->lam", grad, phi) * jac
    tau = h * h / (12.0 * nu)

    def block(la, lc):
        v = np.zeros((b, b))
        v[range(d), range(d)] = nu * K[la, lc]
        v[:d, d] = G[la, :, lc]
        v[d, :d] = -G[lc, :, la]
        v[d, d] = tau * K[la, lc]
        return torch.from_numpy(v).cuda()

    fixed = torch.zeros((g.n, b), dtype=torch.bool, device="cuda")
    fixed[:, :d] = g.boundary[:, None]
    fixed[0, d] = True
    return g, b, [0] * b, g.assemble(b, block, fixed)


def _mhd2d(N, gen, cells=False, decades=3.0):
    """(u, v, p | Bx, By, psi), coupled through a smooth background field; nu and eta log-uniform over
    `decades` below 1, or eta per cell in [1e-4, 1]."""
    g, b, h = _Grid(2, N, "cuda"), 6, 1.0 / N
    nu = 10.0 ** float(-decades * _uniform(gen, 1))
    eta = 10.0 ** (-4.0 * _uniform(gen, N * N)) if cells else 10.0 ** float(-decades * _uniform(gen, 1))
    phi, dphi, pts = _reference_element(2)
    grad, jac = dphi * (2.0 / h), (h / 2.0) ** 2
    K = np.einsum("qla,qma->lm", grad, grad) * jac
    G = -np.einsum("qla,qm->lam", grad, phi) * jac
    tau_p, tau_s = h * h / (12.0 * nu), h * h / (12.0 * eta)
    # B0 = curl of sum c_kl sin(k pi x) sin(l pi y) at the quadrature points
    c = 2.0 * _uniform(gen, 4, 4) - 1.0
    q = torch.from_numpy((pts + 1.0) / 2.0).cuda()
    x = (g.cell[0][:, None] + q[None, :, 0]) * (h * math.pi)
    y = (g.cell[1][:, None] + q[None, :, 1]) * (h * math.pi)
    bx, by = torch.zeros_like(x), torch.zeros_like(x)
    for k in range(1, 5):
        for l in range(1, 5):
            a = c[k - 1, l - 1] / (k * k + l * l)
            bx += a * l * torch.sin(k * x) * torch.cos(l * y)
            by -= a * k * torch.cos(k * x) * torch.sin(l * y)
    s = (bx * bx + by * by).sqrt().max()
    bx, by = bx / s, by / s
    # Y[e, la, a, lc, c] = sum_q curl(phi_la e_a) (phi_lc e_c x B0)_z
    curl = np.stack([-grad[:, :, 1], grad[:, :, 0]], axis=2)
    w = torch.from_numpy(np.einsum("qla,qm->qlam", curl, phi) * jac).cuda()
    Y = torch.stack([(by[:, :, None, None, None] * w[None]).sum(1), (-bx[:, :, None, None, None] * w[None]).sum(1)],
                    dim=4)

    def block(la, lc):
        v = torch.zeros((N * N, b, b), dtype=torch.float64, device="cuda")
        for a in range(2):
            v[:, a, a] = nu * K[la, lc]
            v[:, a, 2] = G[la, a, lc]
            v[:, 2, a] = -G[lc, a, la]
            v[:, 3 + a, 3 + a] = eta * K[la, lc]
            v[:, 3 + a, 5] = G[la, a, lc]
            v[:, 5, 3 + a] = -G[lc, a, la]
        v[:, 2, 2] = tau_p * K[la, lc]
        v[:, 5, 5] = tau_s * K[la, lc]
        v[:, 3:5, 0:2] = Y[:, la, :, lc, :]
        v[:, 0:2, 3:5] = -Y[:, lc, :, la, :].transpose(1, 2)
        return v

    fixed = torch.zeros((g.n, b), dtype=torch.bool, device="cuda")
    fixed[:, [0, 1, 3, 4, 5]] = g.boundary[:, None]
    fixed[0, 2] = True
    return g, b, [0, 0, 0, 1, 1, 1], g.assemble(b, block, fixed)


def _one(case, gen):
    system, N = case["system"], case["N"]
    if system in ("stokes2d", "stokes3d"):
        return _stokes(3 if system == "stokes3d" else 2, N, gen)
    # solves: coefficients within a decade, where every system converges (both near 1e-3 stagnate with this
    # smoother, as the benchmark's batches show)
    return _mhd2d(N, gen, cells=system == "cells", decades=1.0 if case["kind"] in ("solve", "host") else 3.0)


class _System:
    """Device arrays of one system (or batch): row pointers, columns, values, right-hand side."""

    def __init__(self, case, seed):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        self.off = None
        if case["system"] == "q2q1":
            s = problems.mhd2d_q2q1(case["N"], seed)
            self.b, self.fields, self.off = s.b, s.field_of_dof, s.node_field_off
            self.rp, self.ci = torch.from_numpy(s.row_ptr).cuda(), torch.from_numpy(s.col_idx).cuda()
            self.vals = torch.from_numpy(s.vals).cuda()
        elif case["system"] == "batch":
            step = (case["hi"] - case["lo"]) / max(case["nsys"] - 1, 1)
            sizes = [case["lo"] + int(k * step) for k in range(case["nsys"])]
            rp, ci, vals, self.off, nnz = [], [], [], [0], 0
            for N in sizes:
                g, self.b, self.fields, v = _mhd2d(N, gen)
                rp.append(g.rp[:-1] + nnz)
                ci.append(g.ci + self.off[-1])
                vals.append(v)
                nnz += g.ci.numel()
                self.off.append(self.off[-1] + g.n)
            rp.append(torch.tensor([nnz], device="cuda"))
            self.rp, self.ci, self.vals = torch.cat(rp).int(), torch.cat(ci).int(), torch.cat(vals)
        else:
            g, self.b, self.fields, self.vals = _one(case, gen)
            self.rp, self.ci = g.rp.int(), g.ci.int()
        self.n = self.rp.numel() - 1
        self.rhs = 2.0 * _uniform(gen, self.n * self.b) - 1.0


def _params(case):
    p = dict(max_levels=case["levels"], max_coarse=case["max_coarse"], cycle_prec=case["prec"])
    if case["prec"] == 32 and case["system"] in ("stokes3d", "cells"):
        p["coarse_prec"] = 32
    if case["system"] == "cells":
        p.update(mlp=learn.load_weights(), mlp_levels=learn.trained_levels())
    if case["system"] == "q2q1":
        p.update(omega=0.6, sub_solver=2)
    return p


def _solver(case, s, params):
    vals = s.vals.reshape(-1)
    if case["system"] == "batch":
        return bamg.BatchSolver(s.off, s.rp, s.ci, vals, s.b, s.fields, **params)
    if case["system"] == "q2q1":
        return bamg.FieldSolver(s.off, s.rp, s.ci, vals, s.b, **params)
    return bamg.Solver(s.rp, s.ci, vals, s.b, s.fields, **params)


# ---------------------------------------------------------------------------
# the training step's inputs: rows of features and targets, a network in training
# ---------------------------------------------------------------------------
def _training(rows, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    p = torch.from_numpy(np.ascontiguousarray(learn.load_weights(), dtype=np.float32)).cuda()
    ntrain = bamg.MLP_NTRAIN
    p[:ntrain] *= 0.9 + 0.2 * torch.rand(ntrain, device="cuda", generator=gen)
    xm, xs = p[ntrain:ntrain + bamg.NFEAT], p[ntrain + bamg.NFEAT:]
    scale = torch.where(xs != 0, 1.0 / xs, torch.zeros_like(xs))
    x = (xm + scale * torch.randn(rows, bamg.NFEAT, device="cuda", generator=gen)).contiguous()
    t = 0.55 + 0.35 * torch.rand(rows, device="cuda", generator=gen)
    head = torch.randint(0, 2, (rows,), device="cuda", generator=gen, dtype=torch.int32)
    m = 1e-3 * torch.randn(ntrain, device="cuda", generator=gen)
    v = 1e-6 * (0.5 + torch.rand(ntrain, device="cuda", generator=gen))
    return p, x, t, head, m, v


LR, STEP = 2e-3, 400  # the training program's rate, a step well into its first epoch


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case = case
    if case["kind"] == "train":
        st.p, st.x, st.t, st.head, st.m, st.v = _training(case["rows"], seed)
        st.p16 = torch.empty(st.p.numel(), dtype=torch.float16, device="cuda")
        bamg.mlp_pack(st.p, st.p16)
        st.grad = torch.empty(bamg.MLP_NTRAIN, device="cuda")
        st.loss = torch.empty(1, device="cuda")
        return st
    s = st.s = _System(case, seed)
    st.x = torch.zeros_like(s.rhs)
    if case["kind"] == "spmv":
        s.vals = s.vals.reshape(-1)
        return st
    st.params = _params(case)
    if case["kind"] in ("cycle", "solve"):
        st.solver = _solver(case, s, st.params)
        s.vals = None  # the hierarchy holds its own copy
        st.solver.vals = None
    if case["kind"] == "host":
        st.params = bamg.amg_default_params(**st.params)
        host = [t.reshape(-1).cpu().pin_memory() for t in (s.rp, s.ci, s.vals, s.rhs)]
        st.pinned = host + [torch.zeros(s.rhs.numel(), dtype=torch.float64).pin_memory()]
        st.host = [t.numpy() for t in st.pinned]
        s.vals = None
    return st


def _result(st, z):
    return z.float() if st.case["prec"] == 32 else z


def run(st):
    c = st.case
    if c["kind"] == "train":
        bamg.mlp_grad(st.p16, st.x, st.t, st.head, c["rows"], st.grad, st.loss)
        bamg.mlp_adam(st.p, st.p16, st.grad, st.m, st.v, STEP, lr=LR)
        return dict(grad=st.grad, loss=st.loss, params=st.p, params16=st.p16, m=st.m, v=st.v)
    s = st.s
    if c["kind"] == "spmv":
        bamg.bsr_spmv(s.rp, s.ci, s.vals, s.n, s.b, s.rhs, st.x)
        return st.x
    if c["kind"] == "cycle":
        return _result(st, st.solver.apply(s.rhs, st.x))
    if c["kind"] == "setup":
        solver = _solver(c, s, st.params)
        return _result(st, solver.apply(s.rhs, st.x))
    if c["kind"] == "solve":
        st.x.zero_()
        st.solver.solve(s.rhs, st.x, tol=TOL, restart=c["restart"], max_iter=MAX_ITER)
        return st.x
    rp, ci, vals, rhs, x = st.host
    x[:] = 0.0
    bamg.amg_solve_host(rp, ci, vals, s.n, ci.size, s.b, s.fields, rhs, x, tol=TOL, restart=c["restart"],
                        max_iter=MAX_ITER, params=st.params)
    return x


# ---------------------------------------------------------------------------
# work: what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    if case["kind"] == "train":
        n, w = case["rows"], bamg.MLP_NTRAIN
        return dict(bytes=n * (bamg.NFEAT * 4 + 8) + w * 4 * 8, flops=6.0 * n * w)
    if case["system"] == "batch":
        N = (case["lo"] + case["hi"]) / 2.0
        n, nnz, b = case["nsys"] * (N + 1) ** 2, case["nsys"] * (3 * N + 1) ** 2, 6
    elif case["system"] == "q2q1":
        n, nnz, b = (2 * case["N"] + 1) ** 2 + (case["N"] + 1) ** 2, 123.0 * case["N"] ** 2, 3
    else:
        d = 3 if case["system"] == "stokes3d" else 2
        n, nnz = (case["N"] + 1) ** d, (3 * case["N"] + 1) ** d
        b = {"stokes2d": 3, "stokes3d": 4}.get(case["system"], 6)
    m64, vec = nnz * (b * b * 8.0 + 4.0) + 4.0 * n, 8.0 * n * b
    if case["kind"] == "spmv":
        return dict(bytes=m64 + 2 * vec, flops=2.0 * nnz * b * b)
    # a V(1,1) cycle from zero: the pre-smoothing and the residual read one half of the matrix each, the
    # post-smoothing all of it; the coarser levels add about an eighth (2D: a ninth of the nodes, 3D: less)
    mc = nnz * (b * b * case["prec"] / 8.0 + 4.0) + 4.0 * n
    cyc_flops = 4.0 * nnz * b * b * 1.1
    cyc_bytes = mc * 1.1 + 2 * vec
    if case["kind"] == "cycle":
        return dict(bytes=cyc_bytes, flops=cyc_flops)
    if case["kind"] == "setup":
        copies = m64 * 2.1 + (mc if case["prec"] == 32 else 0.0)
        return dict(bytes=copies + cyc_bytes, flops=cyc_flops + 2.0 * nnz * b * b)
    its = {"stokes2d": 60, "stokes3d": 90, "mhd2d": 130}[case["system"]]
    step = dict(bytes=cyc_bytes + m64 + 2 * vec, flops=cyc_flops + 2.0 * nnz * b * b)
    extra = m64 * 2.1 if case["kind"] == "host" else 0.0
    return dict(bytes=its * step["bytes"] + extra, flops=its * step["flops"])


# ---------------------------------------------------------------------------
# exact: the same results in 64 bits, in plain torch and numpy
# ---------------------------------------------------------------------------
def _aggregate(rp, ci):
    """A node that is free with all its neighbours becomes a root (ascending); nodes next to a root join it,
    the others the aggregate with most of their neighbours (ties: the smallest)."""
    n = rp.size - 1
    agg = np.full(n, -1, dtype=np.int64)
    taken = bytearray(n)
    cols, ptr, nc = ci.tolist(), rp.tolist(), 0
    for i in range(n):
        if taken[i]:
            continue
        nb = cols[ptr[i]:ptr[i + 1]]
        if any(taken[j] for j in nb):
            continue
        for j in nb:
            taken[j] = 1
        agg[nb] = nc
        nc += 1
    out = agg.copy()
    for i in np.nonzero(agg < 0)[0]:
        a = agg[ci[rp[i]:rp[i + 1]]]
        a = a[a >= 0]
        out[i] = np.argmax(np.bincount(a))
    return out, nc


def _colours(rp, ci):
    """First fit in ascending node order."""
    n = rp.size - 1
    cols, ptr, col = ci.tolist(), rp.tolist(), [0] * n
    for i in range(n):
        used = 0
        for j in cols[ptr[i]:ptr[i + 1]]:
            if j >= i:
                break
            used |= 1 << col[j]
        c = 0
        while used >> c & 1:
            c += 1
        col[i] = c
    return np.array(col)


class _Exact:
    """The V(1,1) cycle with damped block Gauss-Seidel (omega 0.5), in FP64 on the GPU."""

    def __init__(self, s, levels, max_coarse, omega=0.5):
        self.b, self.F, self.omega = s.b, max(s.fields) + 1, omega
        self.lev = []
        rp, ci, vals = s.rp.long(), s.ci.long(), s.vals.reshape(-1, s.b, s.b)
        b, F = self.b, self.F
        fb = b // F
        while True:
            n = rp.numel() - 1
            row = torch.repeat_interleave(torch.arange(n, device="cuda"), rp.diff())
            L = dict(n=n, row=row, ci=ci, vals=vals)
            self.lev.append(L)
            if len(self.lev) >= levels or n * b <= max_coarse:
                break
            hrp, hci = rp.cpu().numpy(), ci.cpu().numpy()
            agg, nc = _aggregate(hrp, hci)
            if nc in (0, n):
                break
            col = torch.from_numpy(_colours(hrp, hci)).cuda()
            agg = torch.from_numpy(agg).cuda()
            diag = vals[row == ci]
            L["agg"], L["dinv"] = agg, [torch.linalg.inv(diag[:, f * fb:(f + 1) * fb, f * fb:(f + 1) * fb])
                                        for f in range(F)]
            low = col[ci] < col[row]
            L["steps"] = []
            for c in range(int(col.max()) + 1):
                k = (low & (col[row] == c)).nonzero()[:, 0]
                L["steps"].append(((col == c).nonzero()[:, 0], row[k], ci[k], k))
            key, where = torch.unique(agg[row] * nc + agg[ci], return_inverse=True)
            cv = torch.zeros((key.numel(), b, b), dtype=torch.float64, device="cuda").index_add_(0, where, vals)
            rp = torch.zeros(nc + 1, dtype=torch.int64, device="cuda")
            rp[1:] = torch.bincount(key // nc, minlength=nc).cumsum(0)
            ci, vals = key % nc, cv
        # the coarsest matrix: dense, in diagonal blocks where it falls apart (a batch)
        L = self.lev[-1]
        first = torch.arange(L["n"], device="cuda")
        hi = first.clone().scatter_reduce_(0, L["row"], L["ci"], "amax").cpu().numpy()
        reach, cut = 0, [0]
        for i in range(L["n"]):
            if i and reach < i:
                cut.append(i)
            reach = max(reach, int(hi[i]))
        cut.append(L["n"])
        self.coarse = []
        for a, e in zip(cut[:-1], cut[1:]):
            k = ((L["row"] >= a) & (L["row"] < e)).nonzero()[:, 0]
            D = torch.zeros((e - a, b, e - a, b), dtype=torch.float64, device="cuda")
            D[L["row"][k] - a, :, L["ci"][k] - a, :] = L["vals"][k]
            self.coarse.append((a, e, torch.linalg.lu_factor(D.reshape((e - a) * b, (e - a) * b))))

    def _mul(self, L, x):
        out = torch.zeros((L["n"], self.b), dtype=torch.float64, device="cuda")
        for k in range(0, L["ci"].numel(), 1 << 21):
            q = slice(k, k + (1 << 21))
            out.index_add_(0, L["row"][q], torch.bmm(L["vals"][q], x[L["ci"][q]][:, :, None])[:, :, 0])
        return out

    def _smooth(self, L, rhs, x):
        fb = self.b // self.F
        for f in range(self.F):
            d = slice(f * fb, (f + 1) * fb)
            r = (rhs - self._mul(L, x))[:, d].clone()
            t = torch.zeros_like(r)
            for nodes, row, col, k in L["steps"]:
                if k.numel():
                    r.index_add_(0, row, torch.bmm(L["vals"][k][:, d, d], t[col][:, :, None])[:, :, 0], alpha=-1.0)
                t[nodes] = torch.bmm(L["dinv"][f][nodes], r[nodes][:, :, None])[:, :, 0]
            x = x.clone()
            x[:, d] += self.omega * t
        return x

    def cycle(self, rhs, l=0):
        L = self.lev[l]
        if l == len(self.lev) - 1:
            return torch.cat([torch.linalg.lu_solve(*lu, rhs[a:e].reshape(-1, 1)).reshape(-1, self.b)
                              for a, e, lu in self.coarse])
        x = self._smooth(L, rhs, torch.zeros_like(rhs))
        C = self.lev[l + 1]
        rc = torch.zeros((C["n"], self.b), dtype=torch.float64, device="cuda").index_add_(
            0, L["agg"], rhs - self._mul(L, x))
        return self._smooth(L, rhs, x + self.cycle(rc, l + 1)[L["agg"]])


def _exact_training(rows, seed):
    p, x, t, head, m, v = (a.double() if a.is_floating_point() else a.long() for a in _training(rows, seed))
    ntrain, nf, nh, no = bamg.MLP_NTRAIN, bamg.NFEAT, bamg.MLP_H, bamg.MLP_OUT
    q = p.float().half().double()
    w = q[:ntrain].clone().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = (a for a in w.split([nh * nf, nh, nh * nh, nh, no * nh, no]))
    xh = (x - q[ntrain:ntrain + nf]) * q[ntrain + nf:]
    h1 = torch.tanh(xh @ W1.reshape(nh, nf).T + b1)
    h2 = torch.tanh(h1 @ W2.reshape(nh, nh).T + b2)
    y = h2 @ W3.reshape(no, nh).T + b3
    loss = ((y.gather(1, head[:, None])[:, 0] - t) ** 2).mean()
    grad, = torch.autograd.grad(loss, w)
    m, v = 0.9 * m + 0.1 * grad, 0.999 * v + 0.001 * grad * grad
    p = p.clone()
    p[:ntrain] -= LR * (m / (1 - 0.9 ** STEP)) / ((v / (1 - 0.999 ** STEP)).sqrt() + 1e-8)
    return dict(grad=grad, loss=loss.detach().reshape(1), params=p, params16=p, m=m, v=v)


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_training(case["rows"], seed)
    # learned dampings and Schwarz subdomains are the framework's own; an iterate that stops at a tolerance
    # has no value of its own
    if case["kind"] in ("solve", "host") or case["system"] in ("cells", "q2q1"):
        return None
    s = _System(case, seed)
    if case["kind"] == "spmv":
        E = _Exact.__new__(_Exact)
        E.b = s.b
        n = s.n
        L = dict(n=n, ci=s.ci.long(), vals=s.vals.reshape(-1, s.b, s.b),
                 row=torch.repeat_interleave(torch.arange(n, device="cuda"), s.rp.long().diff()))
        return E._mul(L, s.rhs.reshape(n, s.b)).reshape(-1)
    return _Exact(s, case["levels"], case["max_coarse"]).cycle(s.rhs.reshape(s.n, s.b)).reshape(-1)
