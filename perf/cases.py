"""The calls whose speed is measured: what a program that uses this library has it do.

A case is a dict of plain values; `listed()` gives the fixed ones and `draw()`
more of the same ranges. `prepare()` builds on the GPU what the program holds
before the call, `run()` makes the call, `work()` says what it cannot do
without and `exact()` gives its result from plain torch or numpy in 64 bits.

The kinds:
  dot     rbs_exdot: one exact dot on device vectors, from launch-bound lengths
          to ones far beyond L2, well conditioned and with heavy cancellation;
  dots    rbs_exdot_multi with the operand patterns of the solvers' merged
          reductions (k = 2: <r0,r>, <r,r>; k = 5: <r0,r>, <r0,w>, <r0,s>,
          <r0,z>, <r,r>);
  spmv    rbs_spmv_csr on stencil, band and unstructured matrices;
  solve   rbs_solve, classic or pipelined, a bounded number of iterations of a
          system that needs more (so that every pass does the same work);
  batch   rbs_solve_batched on many small to middling convection-diffusion
          systems, classic and pipelined mixed, under the schedule the tuner
          picks for such batches or the default one.
"""
import math
import random

import numpy as np
import torch

import paper_2302_04180_gb300 as rbs

DEV = "cuda"


def listed():
    return [
        # a reduction inside somebody's own small iteration: all latency
        {"name": "dot_64k", "kind": "dot", "n": 1 << 16, "cond": 1e16},
        # an ordinary vector of odd length with heavy cancellation
        {"name": "dot_1m_odd", "kind": "dot", "n": (1 << 20) + 3, "cond": 1e32},
        # long dots, worst and best conditioned: the standalone reduction at stream speed
        {"name": "dot_16m", "kind": "dot", "n": 1 << 24, "cond": 1e48},
        {"name": "dot_128m", "kind": "dot", "n": 1 << 27, "cond": 1.0},
        # the five merged dots of a pipelined iteration, by a program with its own loop
        {"name": "dots5_2m", "kind": "dots", "n": 2000003, "k": 5},
        # one product with the matrices the solvers meet: 7-point, 27-point ...
        {"name": "spmv_poisson128", "kind": "spmv", "matrix": "poisson", "side": 128},
        {"name": "spmv_stencil27_159", "kind": "spmv", "matrix": "stencil27", "side": 159},
        # ... and an unstructured one: ragged rows, some empty, scattered columns
        {"name": "spmv_ragged_500k", "kind": "spmv", "matrix": "ragged", "n": 500003, "max_row": 15},
        # the smallest solve: every step is launch and reduction latency
        {"name": "classic_poisson16", "kind": "solve", "matrix": "poisson", "side": 16, "variant": 0, "iters": 24, "rhs": "ones"},
        # the large solves the library is for, both loops
        {"name": "classic_poisson256", "kind": "solve", "matrix": "poisson", "side": 256, "variant": 0, "iters": 100, "rhs": "ones"},
        {"name": "pipelined_convdiff192", "kind": "solve", "matrix": "convdiff", "side": 192, "variant": 1, "iters": 100, "rhs": "random"},
        # many independent systems at once
        {"name": "batch_512", "kind": "batch", "count": 512, "pattern": 1, "iters": 40, "stepped": True},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["dot", "dot", "dots", "spmv", "spmv", "solve", "solve", "solve", "batch"])
    if kind == "dot":
        return {"kind": kind, "n": int(_log(rng, 1 << 14, 1 << 27)), "cond": rng.choice([1.0, 1e16, 1e32, 1e48])}
    if kind == "dots":
        return {"kind": kind, "n": int(_log(rng, 1 << 15, 1 << 22)), "k": rng.choice([2, 5])}
    if kind == "batch":
        return {"kind": kind, "count": int(_log(rng, 8, 400)), "pattern": rng.randrange(2, 10 ** 6), "iters": rng.randrange(8, 33),
                "stepped": rng.random() < 0.7}
    matrix = rng.choice(["poisson", "convdiff", "stencil27", "banded", "ragged"])
    case = {"kind": kind, "matrix": matrix}
    if matrix in ("poisson", "convdiff"):
        case["side"] = int(_log(rng, 12, 200))
    elif matrix == "stencil27":
        case["side"] = int(_log(rng, 12, 150))
    elif matrix == "banded":
        case["n"], case["band"] = int(_log(rng, 2000, 2e6)), rng.randrange(1, 13)
    else:
        case["n"], case["max_row"] = int(_log(rng, 2000, 1e6)), rng.randrange(3, 40)
    if kind == "solve":
        # diagonally dominant matrices converge in a few iterations: stop earlier still
        case["variant"] = rng.randrange(2)
        case["iters"] = 6 if matrix in ("banded", "ragged") else rng.randrange(10, 1 + min(60, max(10, case["side"])))
        case["rhs"] = rng.choice(["ones", "random"])
    return case


# ---- inputs -------------------------------------------------------------------------


def _gen(seed, tag=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + tag) & 0x7FFFFFFF)
    return g


def _rand(n, g, lo=0.0, hi=1.0):
    return torch.rand(n, dtype=torch.float64, device=DEV, generator=g) * (hi - lo) + lo


def _csr(mask, cols, vals):
    """CSR (int64 rowptr, int32 col, float64 val) from n x k tables of entries; `mask` says which exist."""
    n = mask.shape[0]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(mask.sum(1), 0, out=rowptr[1:])
    return rbs.DeviceCSR(n, rowptr, cols[mask].to(torch.int32), vals[mask])


def _stencil(side, offsets, values):
    """A stencil on a grid of len(offset) dimensions with the outside eliminated, columns ascending."""
    dim = len(offsets[0])
    n = side ** dim
    idx = torch.arange(n, device=DEV)
    coord = [(idx // side ** m) % side for m in range(dim)]
    k = len(offsets)
    mask = torch.empty((n, k), dtype=torch.bool, device=DEV)
    cols = torch.empty((n, k), dtype=torch.int32, device=DEV)
    order = sorted(range(k), key=lambda t: sum(o * side ** m for m, o in enumerate(offsets[t])))
    for j, t in enumerate(order):
        ok = torch.ones(n, dtype=torch.bool, device=DEV)
        for m, o in enumerate(offsets[t]):
            if o:
                ok &= (coord[m] + o >= 0) & (coord[m] + o < side)
        mask[:, j] = ok
        cols[:, j] = (idx + sum(o * side ** m for m, o in enumerate(offsets[t]))).to(torch.int32)
    vals = torch.tensor([values[t] for t in order], dtype=torch.float64, device=DEV).expand(n, k)
    return _csr(mask, cols, vals)


def _star(side, direction, pe):
    """First-order upwind convection-diffusion on 2 or 3 dimensions (pe = 0: Poisson), rows scaled by h^2."""
    dim = len(direction)
    size = math.sqrt(sum(d * d for d in direction))
    p = [pe / (side + 1) * abs(d / size) for d in direction]
    offsets, values = [(0,) * dim], [2.0 * dim + sum(p)]
    for m, d in enumerate(direction):
        for o in (-1, 1):
            offsets.append(tuple(o if i == m else 0 for i in range(dim)))
            values.append(-(1.0 + p[m]) if (o < 0) == (d > 0) and d != 0 else -1.0)
    return _stencil(side, offsets, values)


def _matrix(case, seed):
    kind = case["matrix"]
    if kind == "poisson":
        return _star(case["side"], (1.0, 1.0, 1.0), 0.0)
    if kind == "convdiff":
        return _star(case["side"], (1.0, 1.0, 1.0), 10.0)
    if kind == "stencil27":
        # unsymmetric 27-point model: the neighbours below the centre perturbed
        offsets = [(i, j, k) for k in (-1, 0, 1) for j in (-1, 0, 1) for i in (-1, 0, 1)]
        return _stencil(case["side"], offsets, [26.0 if t == 13 else -0.9999 if t < 13 else -1.0 for t in range(27)])
    if kind == "banded":
        w = case["band"]
        return _stencil(case["n"], [(o,) for o in range(-w, w + 1)],
                        [2.0 * w + 1.0 if o == 0 else -0.9999 if o < 0 else -1.0 for o in range(-w, w + 1)])
    # ragged: up to max_row entries at random columns, one row in twenty empty; for a
    # solve the first entry is a dominant diagonal and no row is empty
    n, k, g = case["n"], case["max_row"], _gen(seed, 3)
    lens = torch.randint(0, k + 1, (n,), device=DEV, generator=g)
    lens[torch.rand(n, device=DEV, generator=g) < 0.05] = 0
    cols = torch.randint(0, n, (n, k), dtype=torch.int32, device=DEV, generator=g)
    vals = _rand(n * k, g, -1.0, 1.0).view(n, k)
    if case["kind"] == "solve":
        lens.clamp_(min=1)
        cols[:, 0] = torch.arange(n, dtype=torch.int32, device=DEV)
        vals[:, 0] = vals.abs().sum(1) + 1.0
    return _csr(torch.arange(k, device=DEV) < lens[:, None], cols, vals)


def _rhs(case, A, seed):
    """b = A x for x a constant or random vector."""
    g = _gen(seed, 5)
    if case["rhs"] == "ones":
        x = _rand(1, g, 0.5, 2.0).expand(A.n).contiguous()
    else:
        x = _rand(A.n, g, -1.0, 1.0)
    return rbs.rbs_spmv_csr(A, x)


def _cancelling(n, cond, seed):
    """Dot operands whose products span 2^0 .. 2^(2b), b = log2(cond)/2, and cancel
    exactly in groups (x, y), (x, -y_hi), (x, -y_lo) and pairs (x, y), (-x, y), but for one
    product u*v about 2 sum|xy| / cond; shuffled. Returns x, y, u*v (exact)."""
    g, h = _gen(seed, 1), random.Random(seed * 31 + 7)
    b = max(1, round(math.log2(cond) / 2))
    trip = (n - 1) // 3
    pair = (n - 1 - 3 * trip) // 2
    m = trip + pair
    one = lambda: (1.0 + _rand(m, g)) * torch.pow(2.0, torch.randint(0, b + 1, (m,), device=DEV, generator=g).double())
    sign = lambda: torch.randint(0, 2, (m,), device=DEV, generator=g).double() * 2.0 - 1.0
    x, y = one() * sign(), one() * sign()
    cut = torch.randint(1, 52, (trip,), device=DEV, generator=g)
    hi = ((y[:trip].view(torch.int64) >> cut) << cut).view(torch.float64)
    xs = [x[:trip], x[:trip], x[:trip], x[trip:], -x[trip:]]
    ys = [y[:trip], -hi, hi - y[:trip], y[trip:], y[trip:]]
    total = 2.0 * float((x[:trip] * y[:trip]).abs().sum()) + 2.0 * float((x[trip:] * y[trip:]).abs().sum())
    e = math.floor(math.log2(2.0 * max(total, 1.0) / cond)) - 50
    u = math.ldexp(h.randrange(1 << 25, 1 << 26), e // 2) * h.choice([-1.0, 1.0])
    v = math.ldexp(h.randrange(1 << 25, 1 << 26), e - e // 2)
    left = n - 1 - 3 * trip - 2 * pair
    xs.append(torch.tensor([u] + [1.5] * left, dtype=torch.float64, device=DEV))
    ys.append(torch.tensor([v] + [0.0] * left, dtype=torch.float64, device=DEV))
    at = torch.randperm(n, device=DEV, generator=g)
    return torch.cat(xs)[at], torch.cat(ys)[at], u * v


def _dot_operands(case, seed):
    if case["cond"] > 2:
        return _cancelling(case["n"], case["cond"], seed)
    g = _gen(seed, 2)
    x, y = (torch.randint(0, 1 << 53, (case["n"],), device=DEV, generator=g).double() * 2.0 ** -53 for _ in range(2))
    return x, y, None


def _dots_operands(case, seed):
    """Vectors as a Krylov loop holds them: entries over a few orders of magnitude."""
    g, n = _gen(seed, 4), case["n"]
    v = [torch.randn(n, dtype=torch.float64, device=DEV, generator=g) * torch.pow(10.0, _rand(n, g, -3.0, 0.0))
         for _ in range(5 if case["k"] == 5 else 2)]
    return ([v[0], v[0], v[0], v[0], v[1]], [v[1], v[2], v[3], v[4], v[1]]) if case["k"] == 5 else ([v[0], v[1]], [v[1], v[1]])


def _batch_shapes(case):
    """(dimension, side) of every system: 1000 to 300000 unknowns, log-uniform, half 2D, half 3D."""
    r = random.Random(case["pattern"])
    out = []
    for _ in range(case["count"]):
        dim = r.choice([2, 3])
        out.append((dim, max(3, round(_log(r, 1000, 300000) ** (1.0 / dim)))))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "dot":
        x, y, _ = _dot_operands(case, seed)
        return {"case": case, "x": x, "y": y}
    if kind == "dots":
        xs, ys = _dots_operands(case, seed)
        return {"case": case, "xs": xs, "ys": ys}
    if kind == "spmv":
        A = _matrix(case, seed)
        return {"case": case, "A": A, "x": _rand(A.n, _gen(seed, 6), -1.0, 1.0)}
    if kind == "solve":
        A = _matrix(case, seed)
        return {"case": case, "A": A, "b": _rhs(case, A, seed), "x": torch.empty(A.n, dtype=torch.float64, device=DEV)}
    shapes, r = _batch_shapes(case), random.Random(seed)
    at, ends = 0, []
    for dim, side in shapes:
        ends.append((at, at + side ** dim))
        at += (side ** dim + 31) // 32 * 32
    x = torch.zeros(at, dtype=torch.float64, device=DEV)
    systems = []
    for k, (dim, side) in enumerate(shapes):
        A = _star(side, tuple(r.uniform(-1.0, 1.0) for _ in range(dim)), r.uniform(0.0, 50.0))
        b = rbs.rbs_spmv_csr(A, torch.ones(A.n, dtype=torch.float64, device=DEV))
        systems.append({"A": A, "b": b, "x": x[ends[k][0]:ends[k][1]], "tol": 1e-14, "maxit": case["iters"], "variant": k % 2})
    return {"case": case, "systems": systems, "x": x}


# ---- the calls ------------------------------------------------------------------------


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "dot":
        return rbs.rbs_exdot(state["x"], state["y"])
    if kind == "dots":
        return rbs.rbs_exdot_multi(state["xs"], state["ys"])
    if kind == "spmv":
        return rbs.rbs_spmv_csr(state["A"], state["x"])
    if kind == "solve":
        r = rbs.rbs_solve(state["A"], state["b"], tol=1e-14, maxit=case["iters"], variant=case["variant"], x_out=state["x"])
        return {"x": r["x"], "hist": r["hist"]}
    got = rbs.rbs_solve_batched(state["systems"], history=False, schedule={"cluster": 0, "split": 0} if case["stepped"] else None)
    return {"x": state["x"], "iters": np.array([r["iters"] for r in got]), "tau": np.array([r["tau_final"] for r in got])}


# ---- what a pass cannot do without ----------------------------------------------------


def _star_nnz(dim, side):
    return side ** dim + 2 * dim * (side - 1) * side ** (dim - 1)


def _size(case):
    """Unknowns and nonzeros (expected, for random rows)."""
    kind = case["matrix"]
    if kind in ("poisson", "convdiff"):
        return case["side"] ** 3, _star_nnz(3, case["side"])
    if kind == "stencil27":
        return case["side"] ** 3, (3 * case["side"] - 2) ** 3
    if kind == "banded":
        w = case["band"]
        return case["n"], (2 * w + 1) * case["n"] - w * (w + 1)
    return case["n"], int(case["n"] * 0.95 * case["max_row"] / 2)


def _solve_work(n, nnz, variant, iters):
    """Per iteration two products (matrix, operand, result and, in the classic loop, the
    dot's other vector) and the vector updates: each vector read or written once a step."""
    vec = 152 if variant == 0 else 304
    return iters * (24 * nnz + (64 if variant == 0 else 48) * n + vec * n), iters * (4 * nnz + (28 if variant == 0 else 58) * n)


def work(case):
    kind = case["kind"]
    if kind == "dot":
        return {"bytes": 16 * case["n"] + 8, "flops": 2 * case["n"]}
    if kind == "dots":
        return {"bytes": 8 * (5 if case["k"] == 5 else 2) * case["n"] + 8 * case["k"], "flops": 2 * case["k"] * case["n"]}
    if kind == "batch":
        total = [0, 0]
        for k, (dim, side) in enumerate(_batch_shapes(case)):
            b, f = _solve_work(side ** dim, _star_nnz(dim, side), k % 2, case["iters"])
            total[0] += b
            total[1] += f
        return {"bytes": total[0], "flops": total[1]}
    n, nnz = _size(case)
    if kind == "spmv":
        return {"bytes": 12 * nnz + 8 * (n + 1) + 16 * n, "flops": 2 * nnz}
    b, f = _solve_work(n, nnz, case["variant"], case["iters"])
    return {"bytes": b, "flops": f}


# ---- results in 64 bits, without the library -------------------------------------------


def _exact_uniform(x, y):
    """Exact dot of vectors of multiples of 2^-53 in [0, 1), rounded once."""
    total, scale = 0, 2.0 ** 53
    for k in range(0, x.numel(), 1 << 24):
        a, b = ((v[k:k + (1 << 24)] * scale).to(torch.int64) for v in (x, y))
        for p, w in (((a >> 27) * (b >> 27), 54), ((a >> 27) * (b & (1 << 27) - 1), 27), ((a & (1 << 27) - 1) * (b >> 27), 27),
                     ((a & (1 << 27) - 1) * (b & (1 << 27) - 1), 0)):
            total += (int((p >> 31).sum()) << (31 + w)) + (int((p & (1 << 31) - 1).sum()) << w)
    return total / (1 << 106)


def _exact_dot(x, y):
    """Products split exactly (Dekker), summed exactly (fsum)."""
    x, y = x.cpu().numpy(), y.cpu().numpy()
    p = x * y

    def halves(a):
        c = a * 134217729.0
        h = c - (c - a)
        return h, a - h

    (xh, xl), (yh, yl) = halves(x), halves(y)
    e = ((xh * yh - p) + xh * yl + xl * yh) + xl * yl
    return math.fsum(np.concatenate([p, e]).tolist())


def _plain(A):
    return torch.sparse_csr_tensor(A.rowptr, A.col.to(torch.int64), A.val, (A.n, A.n))


def _plain_solve(A, b, iters):
    """Textbook Jacobi-preconditioned BiCGStab from zero, plain 64-bit arithmetic."""
    M = _plain(A)
    rows = torch.repeat_interleave(torch.arange(A.n, device=DEV), A.rowptr.diff())
    hit = A.col.to(torch.int64) == rows
    at, diag = rows[hit], A.val[hit]
    first = torch.ones_like(at, dtype=torch.bool)
    first[1:] = at[1:] != at[:-1]  # the first stored (i, i) of a row with several
    d = torch.zeros(A.n, dtype=torch.float64, device=DEV)
    d[at[first]] = diag[first]
    x, r, r0, p = torch.zeros_like(b), b.clone(), b.clone(), b.clone()
    rho = torch.dot(r0, r)
    for _ in range(iters):
        ph = p / d
        s = M @ ph
        alpha = rho / torch.dot(r0, s)
        q = r - alpha * s
        qh = q / d
        y = M @ qh
        omega = torch.dot(q, y) / torch.dot(y, y)
        x = x + alpha * ph + omega * qh
        r = q - omega * y
        new = torch.dot(r0, r)
        p = r + new / rho * (alpha / omega) * (p - omega * s)
        rho = new
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "dot":
        x, y, known = _dot_operands(case, seed)
        return np.array([_exact_uniform(x, y) if known is None else known])
    if kind == "dots":
        xs, ys = _dots_operands(case, seed)
        return np.array([_exact_dot(x, y) for x, y in zip(xs, ys)])
    if kind == "batch":
        return None
    state = prepare(case, seed)
    A = state["A"]
    if kind == "spmv":
        return _plain(A) @ state["x"]
    return {"x": _plain_solve(A, state["b"], case["iters"]), "hist": None}
