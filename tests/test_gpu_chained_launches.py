"""Calls whose kernel starts up while the work before it in the stream ends: the
operands are written right before and overwritten right after each call, eagerly
and in a captured graph with a second stream joined in. Results are compared bit
for bit with the same call on an idle device."""
import pytest

from gpu_common import cuda_device

pytestmark = pytest.mark.gpu

OPS = ["exdot", "multi", "noalloc", "spmv_short", "spmv_long"]


@pytest.fixture(scope="module")
def dev():
    return cuda_device()


def _call(op, dev):
    """(operand, function writing its result for that operand, result)"""
    import torch

    import paper_2302_04180_gb300 as rbs
    from paper_2302_04180_gb300 import gen
    if op.startswith("spmv"):
        A = rbs.to_device(gen.poisson3d(24) if op == "spmv_short" else gen.stencil27(24), dev)
        x = torch.zeros(A.n, dtype=torch.float64, device=dev)
        out = torch.zeros(A.n, dtype=torch.float64, device=dev)
        return x, lambda: rbs.rbs_spmv_csr(A, x, y=out), out
    x = torch.zeros(300001, dtype=torch.float64, device=dev)
    w = torch.linspace(-1.0, 1.0, x.numel(), dtype=torch.float64, device=dev)
    out = torch.zeros(1 if op == "exdot" else 2, dtype=torch.float64, device=dev)
    if op == "exdot":
        return x, lambda: rbs.rbs_exdot(x, w, out=out), out
    if op == "multi":
        return x, lambda: rbs.rbs_exdot_multi([x, x], [w, x], out=out), out
    return x, lambda: rbs.rbs_exdot_noalloc([x, x], [w, x], out), out


@pytest.mark.parametrize("op", OPS)
def test_between_writers(dev, op):
    import torch
    x, call, out = _call(op, dev)
    g = torch.Generator(device=dev).manual_seed(11)
    srcs = [torch.rand(x.numel(), generator=g, dtype=torch.float64, device=dev) - 0.5 for _ in range(6)]
    want = []
    for src in srcs:
        x.copy_(src)
        torch.cuda.synchronize()
        call()
        torch.cuda.synchronize()
        want.append(out.clone())
    got = [torch.empty_like(out) for _ in range(48)]
    for k, t in enumerate(got):
        torch.mul(srcs[k % 6], 1.0, out=x)
        call()
        t.copy_(out)
    torch.cuda.synchronize()
    for k, t in enumerate(got):
        assert torch.equal(t, want[k % 6]), (op, k)


@pytest.mark.parametrize("op", OPS)
def test_in_a_captured_graph(dev, op):
    import torch
    x, call, out = _call(op, dev)
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    src = torch.rand(x.numel(), dtype=torch.float64, device=dev) - 0.5
    half = torch.empty_like(x)
    with torch.cuda.stream(s):
        call()  # the stream's workspace
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    first = torch.empty_like(out)
    with torch.cuda.graph(graph, stream=s):
        other.wait_stream(s)
        with torch.cuda.stream(other):
            torch.mul(src, 0.5, out=half)
        torch.mul(src, 2.0, out=x)
        s.wait_stream(other)
        call()
        first.copy_(out)
        x.add_(half)
        call()
    for _ in range(3):
        src.uniform_(-1.0, 1.0)
        graph.replay()
        torch.cuda.synchronize()
        got = [first.clone(), out.clone()]
        for scaled, t in ((src * 2.0, got[0]), (src * 2.0 + src * 0.5, got[1])):
            x.copy_(scaled)
            torch.cuda.synchronize()
            call()
            torch.cuda.synchronize()
            assert torch.equal(out, t), op
