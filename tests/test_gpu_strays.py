"""Exact dots whose products keep leaving the threads' windows -- some lanes' far
below or above the others', zeros, subnormals, values that rise or fall along the
vectors -- against the oracle, bit for bit, and their time against that of
products that stay: a warp's lanes take the way out of line together."""
import numpy as np
import pytest

from gpu_common import cuda_device, same

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return cuda_device()


@pytest.fixture(scope="module")
def rbs(dev):
    import paper_2302_04180_gb300 as m
    yield m
    for k in ("exdot.grid", "exdot.block"):
        m.rbs_set_param(k, 0)


def _operands(kind, n):
    rng = np.random.default_rng(len(kind) * 1000 + n % 97)
    x, y = rng.uniform(-1.0, 1.0, n), rng.uniform(-1.0, 1.0, n)
    pick = rng.uniform(0.0, 1.0, n)
    if kind == "some_tiny":
        x[pick < 0.01] *= 2.0 ** -400
    elif kind == "few_huge":
        x[pick < 0.001] *= 2.0 ** 300
    elif kind == "spread":
        x *= 2.0 ** rng.uniform(-150.0, 150.0, n)
        y *= 2.0 ** rng.uniform(-150.0, 150.0, n)
    elif kind == "nearly_all_zero":
        x[pick < 0.99] = 0.0
        y[rng.uniform(0.0, 1.0, n) < 0.5] = -0.0
    elif kind == "some_subnormal":
        x[pick < 0.05] *= 2.0 ** -1040
    elif kind == "all_subnormal":
        x *= 2.0 ** -1050
        y *= 2.0 ** -1050
    elif kind == "rise":
        x *= 2.0 ** np.linspace(-900.0, 100.0, n)
    elif kind == "fall":
        x *= 2.0 ** np.linspace(100.0, -900.0, n)
    elif kind == "lowest_window_first":
        # products of 2^-1900 in the first steps, ordinary ones after
        x[: n // 2] *= 2.0 ** -950
        y[: n // 2] *= 2.0 ** -950
    elif kind == "some_infinite":
        x[pick < 0.001] = np.inf
        y = np.abs(y)
    elif kind == "both_infinities":
        x[pick < 0.01] = np.inf
    return x, y


KINDS = ["some_tiny", "few_huge", "spread", "nearly_all_zero", "some_subnormal", "all_subnormal", "rise", "fall",
         "lowest_window_first", "some_infinite", "both_infinities"]


@pytest.mark.parametrize("kind", KINDS)
def test_same_bits_as_the_oracle(rbs, dev, orc, kind):
    """One warp with many steps, a block, and the chosen grid; lengths with and
    without whole steps, odd, and operands off a 16-byte boundary."""
    import torch
    for grid, block, n in ((1, 32, 20001), (1, 32, 383), (3, 64, 50000), (0, 0, (1 << 20) + 3), (0, 0, 4097)):
        rbs.rbs_set_param("exdot.grid", grid)
        rbs.rbs_set_param("exdot.block", block)
        x, y = _operands(kind, n)
        xd, yd = torch.from_numpy(x).to(dev), torch.from_numpy(y).to(dev)
        want = orc.exdot(x, y)
        assert same(rbs.rbs_exdot(xd, yd).item(), want), (kind, grid, block, n)
        got = rbs.rbs_exdot_multi([xd, yd, xd], [yd, yd, xd]).cpu().numpy()
        for g, (a, b) in zip(got, ((x, y), (y, y), (x, x))):
            assert same(g, orc.exdot(a, b)), (kind, grid, block, n)
        assert same(rbs.rbs_exdot(xd[1:], yd[1:]).item(), orc.exdot(x[1:], y[1:])), (kind, n)


# Measured at 2^24: 4.2 and 6.9 times a dot that stays in its windows when each lane went
# out of line by itself, 2.2 and 3.2 since. The bounds are the geometric means.
@pytest.mark.parametrize("kind,times", [("some_tiny", 3.1), ("spread_400", 4.7)])
def test_strays_do_not_hold_the_warp_up_lane_by_lane(rbs, dev, kind, times):
    import torch
    n = 1 << 24
    g = torch.Generator(device=dev)
    g.manual_seed(3)
    rand = lambda: torch.rand(n, dtype=torch.float64, device=dev, generator=g) * 2.0 - 1.0
    x, y, out = rand(), rand(), torch.empty(1, dtype=torch.float64, device=dev)
    if kind == "some_tiny":
        xs, ys = torch.where(rand() < -0.98, x * 2.0 ** -400, x), y
    else:
        two = torch.tensor(2.0, dtype=torch.float64, device=dev)
        xs, ys = x * torch.pow(two, rand() * 100.0), y * torch.pow(two, rand() * 100.0)

    def us(a, b):
        best = []
        for _ in range(7):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            rbs.rbs_exdot(a, b, out)
            e0.record()
            for _ in range(10):
                rbs.rbs_exdot(a, b, out)
            e1.record()
            e1.synchronize()
            best.append(e0.elapsed_time(e1) * 100.0)
        return sorted(best)[3]
    plain, stray = us(x, y), us(xs, ys)
    assert stray < times * plain, (kind, plain, stray)
