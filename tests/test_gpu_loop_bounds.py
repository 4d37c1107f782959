"""The graph loop's own bounds: the largest maxit there is, few iterations again on the
same arguments (the second call runs the graph, whose body then holds no more than
that many), and solves that stop within a body -- converged, at a breakdown,
at a NaN -- on the launch-per-step kernels, against the oracle, bit for bit."""
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
    m.rbs_set_param("vec.block", 0)


@pytest.mark.parametrize("variant", [0, 1])
def test_largest_maxit(rbs, dev, variant):
    import torch
    A = gen.poisson3d(34)  # does not fit one cluster
    Ad = rbs.to_device(A, dev)
    b = rbs.rbs_spmv_csr(Ad, torch.ones(A.n, dtype=torch.float64, device=dev))
    want = rbs.rbs_solve(Ad, b, tol=1e-9, maxit=1000, variant=variant)
    got = rbs.rbs_solve(Ad, b, tol=1e-9, maxit=2 ** 31 - 1, variant=variant, history=False)
    assert want["converged"] == 1 and want["iters"] > 8
    assert (got["converged"], got["iters"]) == (1, want["iters"])
    assert same_array(got["x"].cpu().numpy(), want["x"].cpu().numpy())


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("maxit", [1, 2, 3, 4, 5, 17])
def test_few_iterations_twice(rbs, dev, orc, variant, maxit):
    import torch
    A = gen.poisson3d(34)
    b = gen.random_vector(A.n, 7)
    Ad, bd = rbs.to_device(A, dev), torch.from_numpy(b).to(dev)
    x = torch.empty(A.n, dtype=torch.float64, device=dev)
    o = orc.solve(A, b, tol=1e-14, maxit=maxit, variant=variant)
    for _ in range(3):
        g = rbs.rbs_solve(Ad, bd, tol=1e-14, maxit=maxit, variant=variant, x_out=x)
        assert (g["status"], g["iters"]) == (o["status"], o["iters"]) == (0, maxit)
        assert same_array(g["hist"], o["hist"]) and same_array(x.cpu().numpy(), o["x"])


def _stops():
    """Systems that stop in their first or a later iteration, and how."""
    two = gen.CSR(2, np.array([0, 1, 3], np.int64), np.array([0, 0, 1], np.int32), np.array([1.0, -2.0, 1.0]))
    yield "breakdown", two, np.array([1.0, 1.0]), {}
    n = 1000
    d = gen.CSR(n, np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), 2.0 ** (np.arange(n) % 20 - 10.0))
    yield "one step", d, gen.random_vector(n, 3), {"tol": 1e-14}
    A = gen.poisson3d(5)
    b = gen.random_vector(A.n, 5)
    bad = b.copy()
    bad[7] = np.nan
    yield "nan", A, bad, {}
    # products beyond the range from some iteration on
    yield "overflow", A, b * 2.0 ** 1010, {"tol": 1e-300, "maxit": 40}
    yield "zero", A, np.zeros(A.n), {}
    for k in (1, 2, 3, 5, 6):
        yield f"maxit {k}", A, b, {"tol": 1e-30, "maxit": k}
    for tol in (1e-1, 1e-3, 1e-6, 1e-12):
        yield f"tol {tol}", A, b, {"tol": tol}


# knobs that keep small systems on the launch-per-step kernels
KNOBS = [("spmv.mode", 1), ("spmv.mode", 2), ("spmv.mode", 3), ("vec.block", 256)]


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("knob", KNOBS, ids=lambda k: f"{k[0]}{k[1]}")
def test_stops_on_the_launch_per_step_kernels(rbs, dev, orc, variant, knob):
    import torch
    rbs.rbs_set_param(*knob)
    try:
        for what, A, b, kw in _stops():
            kw = {"tol": 1e-8, "maxit": 60, **kw}
            o = orc.solve(A, b, variant=variant, **kw)
            Ad, bd = rbs.to_device(A, dev), torch.from_numpy(b).to(dev)
            for loop in (rbs.RBS_LOOP_GRAPH, rbs.RBS_LOOP_GRAPH, rbs.RBS_LOOP_HOST):
                g = rbs.rbs_solve(Ad, bd, variant=variant, loop_mode=loop, **kw)
                at = (what, variant, knob, loop)
                assert (g["status"], g["iters"], g["converged"]) == (o["status"], o["iters"], o["converged"]), at
                assert same_array(g["hist"], o["hist"]) and same_array(g["x"].cpu().numpy(), o["x"]), at
    finally:
        rbs.rbs_set_param(knob[0], 0)


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("knob", KNOBS, ids=lambda k: f"{k[0]}{k[1]}")
def test_x0_and_own_diagonal_on_the_launch_per_step_kernels(rbs, dev, orc, variant, knob):
    import torch
    rbs.rbs_set_param(*knob)
    try:
        A = gen.convdiff3d(10, 20.0, (1.0, -0.3, 0.5))
        b, x0 = gen.random_vector(A.n, 4), gen.random_vector(A.n, 5)
        d = gen.random_vector(A.n, 6, lo=4.0, hi=9.0)
        o = orc.solve(A, b, x0=x0, diag=d, tol=1e-9, maxit=400, variant=variant)
        g = rbs.rbs_solve(rbs.to_device(A, dev), torch.from_numpy(b).to(dev), x0=torch.from_numpy(x0).to(dev),
                          jacobi_diag=torch.from_numpy(d).to(dev), tol=1e-9, maxit=400, variant=variant)
        assert (g["status"], g["iters"]) == (o["status"], o["iters"])
        assert same_array(g["hist"], o["hist"]) and same_array(g["x"].cpu().numpy(), o["x"])
    finally:
        rbs.rbs_set_param(knob[0], 0)
