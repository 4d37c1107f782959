"""Solves of matrices with a few very long rows among short ones: the set-up checks
their nonzeros in parallel. Against the oracle, bit for bit, with the errors of the
general set-up; and its time against that of the matrix without them."""
import numpy as np
import pytest

from gpu_common import cuda_device, same_array
from paper_2302_04180_gb300 import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return cuda_device()


@pytest.fixture(scope="module")
def rbs(dev):
    import paper_2302_04180_gb300 as m
    return m


def _arrow(n, rows, length):
    """Tridiagonal but for the given rows, which have `length` nonzeros, the diagonal
    among them."""
    cols = []
    for i in range(n):
        if i in rows:
            c = np.unique(np.concatenate([[i], np.arange(length - 1) * (n // length) % n]))
        else:
            c = np.arange(max(i - 1, 0), min(i + 2, n))
        cols.append(c)
    rowptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
    col = np.concatenate(cols).astype(np.int32)
    val = np.where(col == np.repeat(np.arange(n), np.diff(rowptr)), float(length + 3), -0.5)
    return gen.CSR(n, rowptr, col, val, "arrow")


@pytest.mark.parametrize("length", [255, 256, 257, 258, 3000])
def test_same_bits_and_same_errors(rbs, dev, orc, length):
    import torch
    n = 30011
    A = _arrow(n, {0, n // 2, n - 1}, length)
    b = gen.random_vector(n, 3)
    Ad, bd = rbs.to_device(A, dev), torch.from_numpy(b).to(dev)
    for variant in (0, 1):
        o = orc.solve(A, b, tol=1e-12, maxit=5, variant=variant)
        for loop in (rbs.RBS_LOOP_GRAPH, rbs.RBS_LOOP_HOST):
            g = rbs.rbs_solve(Ad, bd, tol=1e-12, maxit=5, variant=variant, loop_mode=loop)
            assert (g["status"], g["iters"]) == (o["status"], o["iters"])
            assert same_array(g["hist"], o["hist"]) and same_array(g["x"].cpu().numpy(), o["x"])
    row = n // 2
    for what in ("column", "diagonal"):
        B = gen.CSR(n, A.rowptr, A.col.copy(), A.val.copy())
        at = np.arange(A.rowptr[row], A.rowptr[row + 1])
        if what == "column":
            B.col[at[-1]] = n
        else:
            B.val[at[A.col[at] == row]] = 0.0
        with pytest.raises(rbs.RbsError) as e:
            rbs.rbs_solve(rbs.to_device(B, dev), bd, tol=1e-12, maxit=5)
        assert e.value.code == rbs.RBS_EINVAL, what


def test_one_dense_row_does_not_serialise_the_set_up(rbs, dev):
    """Measured: 0.11 ms, 0.09 without the row; 13.8 ms when one thread went through it."""
    import time
    import torch
    n = 200000

    def ms(A):
        Ad, bd = rbs.to_device(A, dev), torch.from_numpy(gen.random_vector(n, 3)).to(dev)
        best = 1e9
        for _ in range(5):
            t = time.perf_counter()
            rbs.rbs_solve(Ad, bd, maxit=0)
            best = min(best, (time.perf_counter() - t) * 1e3)
        return best
    plain = gen.banded(n, 1)
    rowptr = plain.rowptr.copy()
    first = np.arange(n, dtype=np.int32)
    rest = slice(int(rowptr[1]), None)
    rowptr[1:] += n - int(plain.rowptr[1])
    dense = gen.CSR(n, rowptr, np.concatenate([first, plain.col[rest]]).astype(np.int32),
                    np.concatenate([np.full(n, 1e-3), plain.val[rest]]))
    assert ms(dense) < 10.0 * ms(plain)
