"""The bounded wait made to run out inside solves under every row schedule: the
staged short and long rows of the general kernels (spmv.mode 2 and 3, whose exact
windows are then flushed lane by lane) and the diagonal layouts (mode 0), both
loops. Each solve reports RBS_ETIMEOUT, and the next one is right again."""
import numpy as np
import pytest

from gpu_common import cuda_device, same_array
from paper_2302_04180_gb300 import gen

pytestmark = pytest.mark.gpu


MATRICES = {"seven": lambda: gen.poisson3d(24), "twentyseven": lambda: gen.stencil27(19),
            "random": lambda: gen.random_csr(9000, 12, 3, diag_dominant=True)}


# (27 points under mode 2 have no staged chunk, hence no wait)
@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("matrix,mode", [(m, k) for m in MATRICES for k in (0, 2, 3) if (m, k) != ("twentyseven", 2)])
def test_wait_runs_out_in_a_solve(orc, matrix, mode, variant):
    import torch
    dev = cuda_device()
    import paper_2302_04180_gb300 as rbs
    A = MATRICES[matrix]()
    Ad = rbs.to_device(A, dev)
    b = orc.spmv(A, np.ones(A.n))
    bd = torch.from_numpy(b).to(dev)
    o = orc.solve(A, b, tol=1e-8, maxit=6, variant=variant)
    try:
        rbs.rbs_set_param("spmv.mode", mode)
        for loop in (rbs.RBS_LOOP_GRAPH, rbs.RBS_LOOP_HOST):
            rbs.rbs_set_param("test.stall_staging", 1)
            with pytest.raises(rbs.RbsError) as e:
                rbs.rbs_solve(Ad, bd, tol=1e-8, maxit=6, variant=variant, loop_mode=loop)
            assert e.value.code == rbs.RBS_ETIMEOUT
            rbs.rbs_set_param("test.stall_staging", 0)
            g = rbs.rbs_solve(Ad, bd, tol=1e-8, maxit=6, variant=variant, loop_mode=loop)
            assert (g["status"], g["iters"]) == (o["status"], o["iters"])
            assert same_array(g["hist"], o["hist"]) and same_array(g["x"].cpu().numpy(), o["x"])
    finally:
        rbs.rbs_set_param("test.stall_staging", 0)
        rbs.rbs_set_param("spmv.mode", 0)
