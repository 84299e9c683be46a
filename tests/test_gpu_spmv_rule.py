"""bsr_spmv on both sides of the sizes where its row mapping changes, for every
block size, against a product in extended precision."""
import numpy as np
import pytest

from paper_2103_07537_gb300 import bamg, problems as P

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [8192, 65536])
@pytest.mark.parametrize("side", [-1, 0])
@pytest.mark.parametrize("b", [1, 2, 3, 4, 5, 6, 7, 8])
def test_spmv_at_the_mapping_edges(rows, side, b):
    n = -(-rows // b) + side  # the last block row count below, or the first at, the edge
    s = P.random_block_system(int(np.ceil(np.sqrt(n))), b, [0] * b, seed=3 * b + side)
    # the leading n block rows: a ragged last grid line and rows of 4, 6 and 9 blocks
    k = int(s.row_ptr[n])
    rp, ci, va = s.row_ptr[:n + 1].copy(), s.col_idx[:k].copy(), s.vals[:k].copy()
    x = P.uniform_pm1(11, 0, s.n_unknowns)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    y = torch.full((n * b,), np.nan, dtype=torch.float64, device="cuda")
    bamg.bsr_spmv(dev(rp), dev(ci), dev(va.reshape(-1)), n, b, dev(x), y)
    row = np.repeat(np.arange(n), np.diff(rp))
    xl = x.reshape(-1, b).astype(np.longdouble)
    prod = va.astype(np.longdouble) * xl[ci][:, None, :]
    want, mag = np.zeros((n, b), np.longdouble), np.zeros((n, b), np.longdouble)
    np.add.at(want, row, prod.sum(axis=2))
    np.add.at(mag, row, np.abs(prod).sum(axis=2))
    # each entry is a sum of at most 9 b products in some order: |error| <= 9 b u |A| |x| (u = 2^-53)
    err = np.abs(y.cpu().numpy().reshape(n, b) - want)
    assert np.all(err <= 9 * b * 2.0 ** -53 * mag)
