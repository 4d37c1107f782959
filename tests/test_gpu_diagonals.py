"""Solves of matrices laid out by their diagonals against the same solves on the
general row schedules (knob spmv.mode) and the oracle, bit for bit: up to 7 and
up to 32 diagonals, every odd size of the last chunk and odd numbers of
nonzeros, values that start off a 16-byte boundary, matrices whose rows nearly
lie on few diagonals but do not (unsorted or repeated columns, one stray entry
that a sample of rows misses), and batches that mix such systems. Products and
dots are exact chains and sums, so equality is exact."""
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
    yield m
    m.rbs_set_param("spmv.mode", 0)


def _check(rbs, orc, Ad, A, b, iters=6, modes=(0, 2)):
    import torch
    bd = torch.from_numpy(b).cuda()
    for variant in (0, 1):
        o = orc.solve(A, b, tol=1e-13, maxit=iters, variant=variant)
        for mode in modes:
            rbs.rbs_set_param("spmv.mode", mode)
            # the host loop: small systems too take the launch-per-step kernels
            g = rbs.rbs_solve(Ad, bd, tol=1e-13, maxit=iters, variant=variant, loop_mode=rbs.RBS_LOOP_HOST)
            assert (g["status"], g["iters"]) == (o["status"], o["iters"]), (A.name, A.n, variant, mode)
            assert same_array(g["hist"], o["hist"]), (A.name, A.n, variant, mode)
            assert same_array(g["x"].cpu().numpy(), o["x"]), (A.name, A.n, variant, mode)
    rbs.rbs_set_param("spmv.mode", 0)


@pytest.mark.parametrize("band", [0, 1, 3, 4, 8, 12, 15])
def test_bands(rbs, dev, orc, band):
    """1, 3, 7, 9, 17, 25 and 31 diagonals, sizes around chunks of 32 rows and
    around a round of the grid's warps."""
    for n in (40, 63, 64, 65, 1000, 4097):
        A = gen.banded(n, band)
        _check(rbs, orc, rbs.to_device(A, dev), A, gen.random_vector(n, 3 + band))


@pytest.mark.parametrize("make", [lambda: gen.poisson3d(31), lambda: gen.convdiff3d(37, 20.0, (0.3, -1.0, 0.5)),
                                  lambda: gen.convdiff2d(173, 30.0), lambda: gen.stencil27(21), lambda: gen.poisson3d(60)],
                         ids=["p31", "c37", "c2d173", "s21", "p60"])
def test_stencils(rbs, dev, orc, make):
    A = make()
    _check(rbs, orc, rbs.to_device(A, dev), A, orc.spmv(A, np.ones(A.n)), iters=4)


def test_values_off_a_16_byte_boundary(rbs, dev, orc):
    import torch
    A = gen.poisson3d(12)
    Ad = rbs.to_device(A, dev)
    v = torch.empty(A.nnz + 1, dtype=torch.float64, device=dev)
    v[1:] = Ad.val
    Ad.val = v[1:]
    _check(rbs, orc, Ad, A, gen.random_vector(A.n, 5))


@pytest.mark.parametrize("what", ["unsorted", "repeated", "stray", "stray_in_range"])
def test_rows_that_do_not_lie_on_few_diagonals(rbs, dev, orc, what):
    A = gen.poisson3d(20)
    col, val, r = A.col.copy(), A.val.copy(), A.rowptr
    row = 4111
    a, e = r[row], r[row + 1]
    if what == "unsorted":
        col[a:e], val[a:e] = col[a:e][::-1].copy(), val[a:e][::-1].copy()
    elif what == "repeated":
        col[a] = col[a + 1]
    elif what == "stray":
        col[e - 1] = A.n - 3
    else:
        col[a] += 2
    B = gen.CSR(A.n, A.rowptr, col, val, what)
    _check(rbs, orc, rbs.to_device(B, dev), B, gen.random_vector(A.n, 6))


def test_batch_of_both_kinds(rbs, dev, orc):
    """A stepped batch of systems with few diagonals, with many, and with rows that
    do not lie on them, classic and pipelined: each as the oracle has it alone."""
    import torch
    base = gen.poisson3d(17)
    col = base.col.copy()
    col[200] += 1
    mats = [gen.poisson3d(17), gen.CSR(base.n, base.rowptr, col, base.val, "stray"), gen.banded(1500, 9),
            gen.convdiff2d(71, 10.0), gen.random_csr(2500, 9, 3, diag_dominant=True), gen.convdiff3d(23, 30.0),
            gen.banded(33, 2), gen.banded(70001, 3)]
    for rows in (0, 64, 2048):
        systems, want = [], []
        for k, A in enumerate(mats):
            for variant in (0, 1):
                b = gen.random_vector(A.n, 40 + k)
                systems.append({"A": rbs.to_device(A, dev), "b": torch.from_numpy(b).to(dev),
                                "x": torch.zeros(A.n, dtype=torch.float64, device=dev), "tol": 1e-12, "maxit": 5 + k,
                                "variant": variant})
                want.append((A, b, variant, 5 + k))
        got = rbs.rbs_solve_batched(systems, schedule={"cluster": 0, "split": rows})
        for g, (A, b, variant, maxit) in zip(got, want):
            o = orc.solve(A, b, tol=1e-12, maxit=maxit, variant=variant)
            assert (g["status"], g["iters"]) == (o["status"], o["iters"]), (A.name, variant, rows)
            assert same_array(g["hist"], o["hist"]) and same_array(g["x"].cpu().numpy(), o["x"]), (A.name, variant, rows)
