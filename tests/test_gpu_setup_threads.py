"""Setups on two host threads at once, one with large and one with small shared
memory needs of the same kernels: a kernel's shared memory limit belongs to
all threads, so neither setup may lower it for the other.  Every hierarchy's
cycle equals, bit for bit, that of the same setup alone."""
import threading

import numpy as np
import pytest

from paper_2103_07537_gb300 import bamg, problems as P

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def block_diagonal(systems):
    """The systems as one block-diagonal batch."""
    off = np.concatenate([[0], np.cumsum([s.n_nodes for s in systems])])
    nz = np.concatenate([[0], np.cumsum([s.col_idx.size for s in systems])])
    rp = np.concatenate([[0]] + [s.row_ptr[1:] + k for s, k in zip(systems, nz)]).astype(np.int32)
    ci = np.concatenate([s.col_idx + o for s, o in zip(systems, off)]).astype(np.int32)
    return off, rp, ci, np.concatenate([s.vals.reshape(-1) for s in systems])


def maker(kind, large):
    """A function of a stream that sets up one hierarchy: dense inverses in a
    cluster (single systems), per system (batches), or Schwarz factors."""
    kw = dict(max_levels=2, max_coarse=0, autotune=0)
    b = 6 if large else 1
    if kind == "batch":
        ss = [P.random_block_system(n, b, [0] * b, seed=n) for n in ((14, 12) if large else (5, 4))]
        off, *arrays = block_diagonal(ss)
        d = [dev(a) for a in arrays]
        return int(off[-1]) * b, lambda st: bamg.BatchSolver(off, *d, b, [0] * b, stream=st, **kw)
    s = P.random_block_system(24 if large else 9, b, [0] * b, seed=b)
    d = [dev(a) for a in (s.row_ptr, s.col_idx, s.vals.reshape(-1))]
    if kind == "schwarz":
        kw["sub_solver"] = 2
    return s.n_unknowns, lambda st: bamg.Solver(*d, b, s.field_of_dof, stream=st, **kw)


@pytest.mark.parametrize("kind", ["cluster", "batch", "schwarz"])
def test_large_and_small_setups_at_once(kind):
    work = []
    for large in (True, False):
        n, make = maker(kind, large)
        r, stream = dev(np.random.default_rng(n).standard_normal(n)), torch.cuda.Stream()
        torch.cuda.synchronize()
        z = torch.zeros_like(r)
        torch.cuda.synchronize()
        make(stream.cuda_stream).apply(r, z, stream=stream.cuda_stream)
        torch.cuda.synchronize()
        work.append((make, r, stream, z))
    errors = []

    def run(make, r, stream, want):
        try:
            z = torch.zeros_like(r)
            torch.cuda.synchronize()
            for _ in range(150):
                g = make(stream.cuda_stream)
                g.apply(r, z, stream=stream.cuda_stream)
                stream.synchronize()
                assert torch.equal(z.cpu(), want)
                del g
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            errors.append(e)

    threads = [threading.Thread(target=run, args=(m, r, st, z.cpu())) for m, r, st, z in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
