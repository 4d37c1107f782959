"""Small systems solved by one cluster in one launch, against the oracle and
against the launch-per-step loop (loop_mode host), bit for bit: sizes around the
number of CTAs and of threads, the largest systems that fit and the next ones
(which take the other path), ragged and empty rows, wide exponent ranges in the
dots, a system whose nonzeros crowd in few rows, errors and breakdowns. Every
value is exact integers rounded once, so equality is exact."""
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


def _both(rbs, dev, orc, A, b, tol=1e-10, maxit=60, variant=0, **kw):
    import torch
    Ad, bd = rbs.to_device(A, dev), torch.from_numpy(b).to(dev)
    extra = {k: torch.from_numpy(v).to(dev) for k, v in kw.items()}
    o = orc.solve(A, b, tol=tol, maxit=maxit, variant=variant, x0=kw.get("x0"), diag=kw.get("jacobi_diag"))
    for loop in (rbs.RBS_LOOP_GRAPH, rbs.RBS_LOOP_HOST):
        g = rbs.rbs_solve(Ad, bd, tol=tol, maxit=maxit, variant=variant, loop_mode=loop, **extra)
        what = (A.name, A.n, variant, loop)
        assert (g["status"], g["iters"], g["converged"]) == (o["status"], o["iters"], o["converged"]), what
        assert same_array(g["hist"], o["hist"]), what
        assert same_array(g["x"].cpu().numpy(), o["x"]), what
        assert same_array([g["tau0"], g["tau_max"], g["tau_final"]], [o["tau0"], o["tau_max"], o["tau_final"]]), what
    return o


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 33, 511, 513, 8191, 8193])
def test_sizes(rbs, dev, orc, n, variant):
    A = gen.banded(n, 2) if n > 4 else gen.banded(n, 1)
    _both(rbs, dev, orc, A, gen.random_vector(n, 4), variant=variant)


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("make", [lambda: gen.poisson3d(23), lambda: gen.poisson3d(24), lambda: gen.poisson3d(27),
                                  lambda: gen.poisson3d(28), lambda: gen.stencil27(13), lambda: gen.stencil27(20),
                                  lambda: gen.convdiff2d(101, 20.0), lambda: gen.convdiff3d(20, 40.0, (1.0, -0.3, 0.2))],
                         ids=["p23", "p24", "p27", "p28", "s13", "s20", "c101", "c20"])
def test_stencils_up_to_and_past_what_fits(rbs, dev, orc, make, variant):
    A = make()
    _both(rbs, dev, orc, A, orc.spmv(A, np.ones(A.n)), maxit=25, variant=variant)


@pytest.mark.parametrize("variant", [0, 1])
def test_ragged_rows_and_own_diagonal(rbs, dev, orc, variant):
    A = gen.random_csr(3001, 20, 5, dup_frac=0.2, diag_dominant=True)
    _both(rbs, dev, orc, A, gen.random_vector(A.n, 3), variant=variant)
    B = gen.random_csr(2000, 9, 6, empty_frac=0.3)
    d = 1.0 + gen.random_vector(B.n, 8, lo=0.0, hi=1.0)
    _both(rbs, dev, orc, B, gen.random_vector(B.n, 9), variant=variant, maxit=12, jacobi_diag=d,
          x0=gen.random_vector(B.n, 10))


@pytest.mark.parametrize("variant", [0, 1])
def test_crowded_rows_take_the_other_path(rbs, dev, orc, variant):
    """All off-diagonal entries in the first rows: one CTA's share would not fit."""
    n, k = 6000, 600
    rows = [np.concatenate([[i], np.setdiff1d(np.arange(k) * 9 + i % 7, [i])]) if i < 150 else np.array([i])
            for i in range(n)]
    rowptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    col = np.concatenate(rows).astype(np.int32)
    val = gen.random_vector(col.size, 11)
    val[rowptr[:-1]] = 700.0
    _both(rbs, dev, orc, gen.CSR(n, rowptr, col, val, "crowded"), gen.random_vector(n, 12), variant=variant)


@pytest.mark.parametrize("variant", [0, 1])
def test_wide_exponents(rbs, dev, orc, variant):
    """Right-hand sides over 600 decades, scattered or falling along the rows, so
    that the CTAs' partial sums lie far apart or span more limbs than travel by mail."""
    A = gen.poisson3d(14)
    e = gen.random_vector(A.n, 13, lo=-140.0, hi=140.0)
    _both(rbs, dev, orc, A, gen.random_vector(A.n, 14) * 10.0 ** e, variant=variant, maxit=8)
    fall = 10.0 ** np.linspace(140.0, -140.0, A.n)
    _both(rbs, dev, orc, A, gen.random_vector(A.n, 15) * fall, variant=variant, maxit=8)
    zero = np.zeros(A.n)
    zero[A.n // 2] = 1.0
    _both(rbs, dev, orc, A, zero, variant=variant, maxit=20)


@pytest.mark.parametrize("variant", [0, 1])
def test_errors_and_ends(rbs, dev, orc, variant):
    import torch
    A = gen.poisson3d(9)
    b = orc.spmv(A, np.ones(A.n))
    for maxit, tol in ((0, 1e-8), (1, 1e-30), (500, 1e-12)):
        _both(rbs, dev, orc, A, b, tol=tol, maxit=maxit, variant=variant)
    _both(rbs, dev, orc, A, np.zeros(A.n), variant=variant)
    bad = b.copy()
    bad[17] = np.inf
    assert rbs.rbs_solve(rbs.to_device(A, dev), torch.from_numpy(bad).to(dev), variant=variant)["status"] == rbs.RBS_ENAN
    xs = torch.full((A.n,), 7.0, dtype=torch.float64, device=dev)
    for what in ("col", "rowptr", "end", "diag"):
        B = gen.CSR(A.n, A.rowptr.copy(), A.col.copy(), A.val.copy())
        if what == "col":
            B.col[100] = A.n
        elif what == "rowptr":
            B.rowptr[50] = B.rowptr[52]
        elif what == "end":
            B.rowptr[-1] -= 1
        else:
            B.val[(B.col == 5) & (np.repeat(np.arange(A.n), np.diff(A.rowptr)) == 5)] = 0.0
        Bd = rbs.to_device(B, dev)
        with pytest.raises(rbs.RbsError) as e:
            rbs.rbs_solve(Bd, torch.from_numpy(b).to(dev), variant=variant, x_out=xs)
        assert e.value.code == rbs.RBS_EINVAL, what
        assert (xs == 7.0).all(), what
