"""Host code of the library against a fake CUDA runtime (host_library.py): what it
allocates, copies and launches where no GPU is needed to tell right from wrong."""
import numpy as np
import pytest

from host_library import host_library
from paper_2302_04180_gb300 import gen


@pytest.fixture()
def host():
    with host_library() as h:
        yield h
        assert h.faults() == ""


def _system(h, A, maxit, variant=0):
    return {"A": h.csr(A), "b": h.device(np.ones(A.n)), "x": h.device(np.zeros(A.n)), "tol": 1e-8, "maxit": maxit,
            "variant": variant}


def test_stepped_batch_reads_the_schedule_knob_once(host):
    """spmv.mode changed by another thread while a stepped batch is being laid out: the
    systems' layouts by diagonals lie in the memory that was sized for them."""
    A = gen.poisson3d(20)
    systems = [_system(host, A, 3, v) for v in (0, 1)]
    host.rbs.rbs_stream_status()  # the workspace exists
    host.rbs.rbs_set_param("spmv.mode", 2)
    stray = []

    def change(call, what, n):
        if call == "cudaMalloc":
            host.rbs.rbs_set_param("spmv.mode", 0)
        if call == "launch" and "k_step_prepare" in what:
            stray.append(host.fake.fake_stray_pointers())
    host.fail = change
    try:
        host.rbs.rbs_solve_batched(systems, schedule={"cluster": 0, "split": 0})
    finally:
        host.fail = None
        host.rbs.rbs_set_param("spmv.mode", 0)
    assert len(stray) == 2 and not any(stray)


def _diagonal(n):
    return gen.CSR(n, np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), np.ones(n))


@pytest.mark.parametrize("sizes", [(1867776, 1088), (3735552, 70000, 900)])
def test_stepped_batch_task_list_may_grow(host, sizes):
    """Rows per block follow the rows still iterating, in steps of 64: once the small
    system has run its iterations the large one may take more blocks than both did."""
    systems = [_system(host, _diagonal(n), 20 if k == 0 else 3) for k, n in enumerate(sizes)]
    got = host.rbs.rbs_solve_batched(systems, history=False, schedule={"cluster": 0, "split": 0})
    assert len(got) == len(sizes) and host.faults() == ""


NO_MEMORY, CLUSTER_FAILED = 2, 912  # cudaErrorMemoryAllocation, cudaErrorClusterOutOfResources


def _solve(host, A, **kw):
    return host.rbs.rbs_solve(host.csr(A), host.device(np.ones(A.n)), tol=1e-8, maxit=20, x_out=host.device(np.zeros(A.n)), **kw)


@pytest.mark.parametrize("variant", [0, 1])
def test_small_solve_goes_on_when_its_launch_is_refused(host, variant):
    """A refused cluster launch is no error of the solve: the launch-per-step loop runs it."""
    A = gen.poisson3d(8)
    host.fail = lambda call, what, n: CLUSTER_FAILED if call == "launch" and "k_small" in what else 0
    _solve(host, A, variant=variant)
    host.fail = None
    names = " ".join(host.launched())
    assert "k_small" in names and ("k_cls_k1" if variant == 0 else "k_pipe_p1") in names
    host.events.clear()
    _solve(host, A, variant=variant)  # nothing of the refusal is left
    assert [n for n in host.launched() if "k_small" in n] and not [n for n in host.launched() if "k_prepare" in n]


def _sizes(host):
    return {n for call, _, n in host.events if call == "cudaMalloc"}


def test_solve_goes_on_without_room_for_the_layout(host):
    """The diagonal layout is scratch that a solve can do without: when it does not fit,
    the general rows run, and nothing of the refusal is left."""
    A = gen.poisson3d(34)
    host.rbs.rbs_set_param("spmv.mode", 2)
    _solve(host, A)
    host.rbs.rbs_set_param("spmv.mode", 0)
    needed = _sizes(host)
    host.rbs.rbs_release()
    host.events.clear()
    host.fail = lambda call, what, n: NO_MEMORY if call == "cudaMalloc" and n not in needed else 0
    _solve(host, A)
    assert _sizes(host) - needed, "nothing was refused"
    k1 = [n for n in host.launched() if "k_cls_k1" in n]
    assert k1 and all("Lin" not in n for n in k1), k1  # (a negative template argument is a diagonal kernel)
    host.fail = None
    host.events.clear()
    _solve(host, A)
    assert [n for n in host.launched() if "k_cls_k1" in n and "Lin7E" in n]


def test_stepped_batch_goes_on_without_room_for_the_layouts(host):
    A = gen.poisson3d(20)
    systems = [_system(host, A, 3, v) for v in (0, 1)]

    def run():
        host.events.clear()
        host.rbs.rbs_solve_batched(systems, schedule={"cluster": 0, "split": 0})
    host.rbs.rbs_set_param("spmv.mode", 2)
    run()
    host.rbs.rbs_set_param("spmv.mode", 0)
    needed = _sizes(host)
    host.rbs.rbs_release()
    host.fail = lambda call, what, n: NO_MEMORY if call == "cudaMalloc" and n not in needed else 0
    run()
    assert _sizes(host) - needed, "nothing was refused"
    assert [n for n in host.launched() if "k_step_cls_k1" in n] and host.fake.fake_stray_pointers() == 0
    host.fail = None
    run()
    assert host.fake.fake_stray_pointers() == 0


def test_diagonal_product_runs_at_the_carveout_of_its_own_solve(host):
    """smem.carveout changed and changed back between solves: the split that k_spmv_diag
    runs at is the one its grid was sized for."""
    A = gen.poisson3d(34)
    before = host.rbs.rbs_get_param("smem.carveout")
    try:
        for c in (61, 0, 61, 62, 0):  # (61 and 62: values that no other test of this process applies)
            host.rbs.rbs_set_param("smem.carveout", c)
            _solve(host, A, variant=1)
            seen = last = None
            for call, what, n in host.events:
                if call == "carveout" and "k_spmv_diagILi7E" in what:
                    seen = n
                if call == "launch" and "k_spmv_diagILi7E" in what:
                    last = seen
            assert last == c, (c, last)
    finally:
        host.rbs.rbs_set_param("smem.carveout", before)


def test_server_admits_without_looking_for_layouts(host):
    """A served system has no room for a layout by diagonals: its admission does not
    launch the kernel that samples them; a stepped batch's does."""
    A = gen.poisson3d(9)
    srv = host.rbs.RbsServer(engines=1, max_active=4)
    tickets = [srv.submit(_system(host, A, 3, v)) for v in (0, 1)]
    for t in tickets:
        assert srv.wait(t)["status"] == 0
    srv.close()
    assert [n for n in host.launched() if "k_step_prepare" in n]
    assert not [n for n in host.launched() if "k_step_sample" in n]
    host.rbs.rbs_solve_batched([_system(host, A, 2)], schedule={"cluster": 0, "split": 0})
    assert [n for n in host.launched() if "k_step_sample" in n]
