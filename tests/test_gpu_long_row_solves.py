"""Whole histories through the long-row kernels (spmv.mode 3: the fused K1/K3 and the
product that keep rows in registers), which matrices of few diagonals no longer take
by themselves, and the diagonal layout of more than seven over several rounds of its
tiles. Against the oracle, bit for bit."""
import numpy as np
import pytest

from gpu_common import cuda_device, same_array
from paper_2302_04180_gb300 import gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("side,mode,maxit", [(40, 3, 800), (80, 0, 3), (80, 3, 3)],
                         ids=["long_rows_40", "tiles_80", "long_rows_80"])
def test_27_points(orc, side, mode, maxit, variant):
    import torch
    dev = cuda_device()
    import paper_2302_04180_gb300 as rbs
    A = gen.stencil27(side)
    b = orc.spmv(A, np.ones(A.n))
    o = orc.solve(A, b, tol=1e-10, maxit=maxit, variant=variant)
    try:
        rbs.rbs_set_param("spmv.mode", mode)
        g = rbs.rbs_solve(rbs.to_device(A, dev), torch.from_numpy(b).to(dev), tol=1e-10, maxit=maxit, variant=variant)
    finally:
        rbs.rbs_set_param("spmv.mode", 0)
    assert g["iters"] == o["iters"] and g["status"] == o["status"] == 0
    assert same_array(g["hist"], o["hist"]) and same_array(g["x"].cpu().numpy(), o["x"])
