"""The shared-memory windows of the standalone exact dot where they can go
wrong, bit for bit against the oracle: carries that leave a product's five
words, products above and below the window, zeros, subnormals and non-finite
operands among ordinary products, and lengths around the steps of the loop.
The values are exact sums rounded once, so equality is exact."""
import numpy as np
import pytest

from gpu_common import bits, cuda_device, same
from paper_2302_04180_gb300 import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return cuda_device()


@pytest.fixture(scope="module")
def rbs(dev):
    import paper_2302_04180_gb300 as m
    yield m
    for k in ("exdot.grid", "exdot.block", "exdot.window"):
        m.rbs_set_param(k, 0)


def _check(rbs, dev, orc, x, y, what):
    import torch
    xt, yt = torch.from_numpy(x).to(dev), torch.from_numpy(y).to(dev)
    ref = orc.exdot(x, y)
    for window in (0, 1, 2):
        for grid, block in ((1, 32), (0, 0)):
            rbs.rbs_set_param("exdot.window", window)
            rbs.rbs_set_param("exdot.grid", grid)
            rbs.rbs_set_param("exdot.block", block)
            got = rbs.rbs_exdot(xt, yt).item()
            assert same(got, ref), (what, window, grid, got, ref)


ONES = 2.0 - 2.0 ** -52  # a significand of 53 ones: its square has 52 ones in a row


def _steps(rng, kind):
    """One product per step; with one warp every thread sees these in order."""
    if kind == "carry":
        # words of all ones, then products whose top word lands on them
        return [(ONES * 2.0 ** (e // 2), ONES * 2.0 ** (e - e // 2)) for e in (0, 57, 89, 121, 31, 63, 95, 0, 1, 30)] * 3
    if kind == "carry_signs":
        return [(s * ONES * 2.0 ** (e // 2), ONES * 2.0 ** (e - e // 2))
                for e in (0, 57, 89, 31, 63) for s in (1.0, -1.0, 1.0)]
    if kind == "climb":
        return [(ONES * 2.0 ** e, 1.0 + 2.0 ** -50) for e in range(-1000, 1000, 61)]
    if kind == "fall":
        return [(ONES * 2.0 ** e, -1.0 - 2.0 ** -50) for e in range(1000, -1000, -61)]
    if kind == "zeros":
        return [(1.5, 2.5), (0.0, 3.0), (-0.0, 1e300), (4.0, 0.0), (1e-300, -0.0), (0.0, 0.0), (-3.25, 1e-5)] * 4
    if kind == "zeros_first":
        return [(0.0, 1.0)] * 9 + [(3.0, 7.0), (0.0, 2.0), (1e-200, 1e-100)]
    if kind == "subnormal":
        return [(2.0 ** -1074, 1.0), (3.0 * 2.0 ** -1074, 2.0 ** 1000), (1.0, 1.0), (2.0 ** -1060, -(2.0 ** -1060)),
                (2.0 ** -1074, 2.0 ** -1074)]
    if kind == "nonfinite":
        return [(1.0, 2.0), (np.inf, 2.0), (0.0, 5.0), (1e-300, 1e-300)]
    if kind == "nan":
        return [(1.0, 2.0), (0.0, np.inf), (3.0, 4.0)]
    return [(float(rng.uniform(-1, 1) * 2.0 ** rng.uniform(-500, 500)), float(rng.uniform(-1, 1) * 2.0 ** rng.uniform(-500, 500)))
            for _ in range(40)]


@pytest.mark.parametrize("kind", ["carry", "carry_signs", "climb", "fall", "zeros", "zeros_first", "subnormal",
                                  "nonfinite", "nan", "wild"])
def test_products_in_every_place(rbs, dev, orc, kind):
    rng = np.random.default_rng(5)
    steps = _steps(rng, kind)
    x = np.concatenate([np.full(64, s[0]) for s in steps])
    y = np.concatenate([np.full(64, s[1]) for s in steps])
    _check(rbs, dev, orc, x, y, kind)
    at = rng.permutation(x.size)  # lanes of a warp in different places
    _check(rbs, dev, orc, np.ascontiguousarray(x[at]), np.ascontiguousarray(y[at]), kind + " shuffled")


def test_lengths_around_the_loop_steps(rbs, dev, orc):
    """Two blocks of 32 threads step over 128 elements at a time, two pairs per
    turn: every length up to five turns' edges, odd ones and remainders."""
    import torch
    x, y, _ = gen.ill_conditioned_dot(1400, 1e24, 3)
    xt, yt = torch.from_numpy(x).to(dev), torch.from_numpy(y).to(dev)
    rbs.rbs_set_param("exdot.grid", 2)
    rbs.rbs_set_param("exdot.block", 32)
    try:
        for n in sorted({m * 128 + d for m in range(11) for d in (-1, 0, 1, 2, 3, 65) if m * 128 + d >= 0}):
            got = rbs.rbs_exdot(xt[:n], yt[:n]).item()
            assert same(got, orc.exdot(x[:n], y[:n])), n
    finally:
        rbs.rbs_set_param("exdot.grid", 0)
        rbs.rbs_set_param("exdot.block", 0)


def test_several_dots_in_one_launch(rbs, dev, orc):
    """1 to 6 dots of mixed ranges, aligned and unaligned operands side by side."""
    import torch
    n = 50001
    vs = [gen.random_vector(n + 1, 21, t) * 10.0 ** gen.random_vector(n + 1, 21, t + 50, -60, 60) for t in range(4)]
    ts = [torch.from_numpy(v).to(dev) for v in vs]
    for k in range(1, 7):
        ops = [(j % 4, (j * 3 + 1) % 4, j & 1) for j in range(k)]
        out = rbs.rbs_exdot_multi([ts[a][o:n + o] for a, _, o in ops], [ts[b][:n] for _, b, _ in ops]).cpu().numpy()
        ref = [orc.exdot(np.ascontiguousarray(vs[a][o:n + o]), np.ascontiguousarray(vs[b][:n])) for a, b, o in ops]
        assert (bits(out) == bits(ref)).all(), k
