"""The products, refreshes and sums that users of this library run, as measurable cases.

``listed()`` names one case per kind of use, ``draw()`` gives further ones of the
same ranges; ``prepare()`` builds a case's matrices on the GPU together with the
handle that a program keeps, and ``run()`` is one pass through the public entry
points.  A case fixes its matrices' sparsity patterns (so the sizes of its
results), the seed draws their values.

Ranges: grids of 100 to 1,000,000 nodes with 5-, 9-, 7- and 27-point operators;
random rows of 3 to 40 entries (the row lengths of the batched workload) in
matrices of 100 to 200,000 rows; R-MAT graphs of scale 10 to 18 with 16 edges
per vertex; batches of 8 to 256 uneven pairs of 100 to 50,000 rows.
"""
import math

import numpy as np
import torch

from paper_2103_11991_gb300 import spgemm as K

DEVICE = "cuda"
RMAT = (0.57, 0.19, 0.19)


# ----------------------------------------------------------------------------
# The cases
# ----------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a 2D Laplacian squared, latency as the caller sees it
        {"name": "laplace2d_64", "op": "product", "kind": "grid", "dims": "64x64", "points": 5, "arith": 0},
        # one small product of unstructured rows, as in a loop over many small systems
        {"name": "random_3001", "op": "product", "kind": "random", "rows": 3001, "inner": 3001, "cols": 3001,
         "low": 3, "high": 40, "unsorted": False, "pattern": 1, "arith": 0},
        # a 3D finite-element operator squared in native float64
        {"name": "stencil27_100", "op": "product", "kind": "grid", "dims": "100x100x100", "points": 27, "arith": 1},
        # the same kind of operator on a ragged grid with new values on a known structure: numeric phase alone
        {"name": "stencil27_refresh", "op": "refresh", "kind": "grid", "dims": "61x53x47", "points": 27, "arith": 0},
        # the AMG triple product R (A P) of a 7-point Laplacian and 2x2x2 aggregates
        {"name": "galerkin_128", "op": "galerkin", "dims": "128x128x128"},
        # AMG prolongator smoothing (I - omega D^-1 A) P on a ragged grid
        {"name": "jacobi_ragged", "op": "jacobi", "dims": "121x97x133", "omega": 2.0 / 3.0},
        # the sum of two large matrices of random rows
        {"name": "spadd_500k", "op": "spadd", "rows": 500000, "cols": 500000, "low": 30, "high": 30,
         "unsorted": False, "pattern": 31, "alpha": 1.5, "beta": -0.5},
        # the square of a power-law graph, rows of 1 to 10^5 entries
        {"name": "rmat_18", "op": "product", "kind": "rmat", "scale": 18, "pattern": 20, "arith": 0},
        # the learned one-pass form on a smaller graph, rows sized by their flop bound
        {"name": "learned_rmat_15", "op": "learned", "kind": "rmat", "scale": 15, "pattern": 21, "arith": 0},
        # rectangular product whose rows are stored in no order, as assembled by an application
        {"name": "random_unsorted", "op": "product", "kind": "random", "rows": 100003, "inner": 80021,
         "cols": 60013, "low": 3, "high": 40, "unsorted": True, "pattern": 2, "arith": 0},
        # many uneven independent products in one call
        {"name": "batch_256", "op": "batch", "count": 256, "rows_low": 100, "rows_high": 50000, "mix": 5000},
        # gradient of the row-capacity network on one training batch (the trainer's default size)
        {"name": "mlp_grad_4096", "op": "mlp_grad", "samples": 4096},
    ]


def _log_uniform(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def _draw_dims(rng, low, high, nd):
    """A ragged grid of about a log-uniform number of nodes, at least 3 per side."""
    nodes = math.exp(rng.uniform(math.log(low), math.log(high)))
    side = nodes ** (1.0 / nd)
    dims = []
    for _ in range(nd - 1):
        dims.append(max(3, int(round(side * rng.uniform(0.7, 1.4)))))
    dims.append(max(3, int(nodes / math.prod(dims))))
    return "x".join(str(d) for d in dims)


def _draw_grid(rng, high):
    points = rng.choice([5, 9, 7, 27])
    return {"kind": "grid", "dims": _draw_dims(rng, 100, high, 2 if points in (5, 9) else 3), "points": points}


def _draw_random(rng):
    rows, inner, cols = (_log_uniform(rng, 100, 200000) for _ in range(3))
    low = rng.randint(3, 20)
    return {"kind": "random", "rows": rows, "inner": inner, "cols": cols, "low": low,
            "high": rng.randint(low, 40), "unsorted": rng.random() < 0.25, "pattern": rng.randint(0, 1 << 20)}


def _draw_operands(rng, scale):
    kind = rng.choice(["grid", "random", "rmat"])
    if kind == "grid":
        return _draw_grid(rng, 900000)
    if kind == "random":
        return _draw_random(rng)
    return {"kind": "rmat", "scale": rng.randint(10, scale), "pattern": rng.randint(0, 1 << 20)}


def draw(rng):
    op = rng.choice(["product", "product", "product", "refresh", "galerkin", "jacobi", "spadd", "learned", "batch",
                     "mlp_grad"])
    if op in ("product", "refresh", "learned"):
        return {"op": op, **_draw_operands(rng, 17 if op == "product" else 16), "arith": rng.choice([0, 0, 1])}
    if op == "galerkin":
        return {"op": op, "dims": _draw_dims(rng, 1000, 2000000, 3)}
    if op == "jacobi":
        return {"op": op, "dims": _draw_dims(rng, 1000, 2000000, 3), "omega": round(rng.uniform(0.5, 1.0), 3)}
    if op == "spadd":
        low = rng.randint(3, 30)
        return {"op": op, "rows": _log_uniform(rng, 1000, 500000), "cols": _log_uniform(rng, 1000, 500000),
                "low": low, "high": rng.randint(low, 40), "unsorted": rng.random() < 0.25,
                "pattern": rng.randint(0, 1 << 20), "alpha": round(rng.uniform(-2, 2), 3),
                "beta": round(rng.uniform(-2, 2), 3)}
    if op == "batch":
        return {"op": op, "count": _log_uniform(rng, 8, 200), "rows_low": 100,
                "rows_high": _log_uniform(rng, 2000, 50000), "mix": rng.randint(0, 1 << 20)}
    return {"op": op, "samples": _log_uniform(rng, 1000, 200000)}


# ----------------------------------------------------------------------------
# Matrices: (m, n, rowptr int32, colind int32, vals float64), all on the GPU
# ----------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))
    return g


def _uniform(g, count, low, high):
    return torch.rand(count, generator=g, device=DEVICE, dtype=torch.float64) * (high - low) + low


def _from_keys(m, n, keys):
    """rowptr and colind of sorted keys row * n + col."""
    rows = torch.div(keys, n, rounding_mode="floor")
    rowptr = torch.zeros(m + 1, dtype=torch.int64, device=DEVICE)
    torch.cumsum(torch.bincount(rows, minlength=m), 0, out=rowptr[1:])
    return rowptr.to(torch.int32), (keys - rows * n).to(torch.int32)


def _dims(case):
    return [int(d) for d in case["dims"].split("x")]


def _offsets(points):
    """Grid offsets (x first), ascending in the linear index of the node."""
    if points == 5:
        return [(0, -1), (-1, 0), (0, 0), (1, 0), (0, 1)]
    if points == 9:
        return [(x, y) for y in (-1, 0, 1) for x in (-1, 0, 1)]
    if points == 7:
        return [(0, 0, -1), (0, -1, 0), (-1, 0, 0), (0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)]
    return [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]


def _grid(dims, points, g):
    """Operator with variable coefficients: off-diagonal entries in [-1.5, -0.5), the
    diagonal as large as the number of neighbours, plus the cell's own share."""
    offsets = _offsets(points)
    count = math.prod(dims)
    node = torch.arange(count, device=DEVICE)
    at, stride, strides = [], 1, []
    for d in dims:
        at.append(torch.div(node, stride, rounding_mode="floor") % d)
        strides.append(stride)
        stride *= d
    cols = torch.empty((count, len(offsets)), dtype=torch.int32, device=DEVICE)
    inside = torch.ones((count, len(offsets)), dtype=torch.bool, device=DEVICE)
    for k, o in enumerate(offsets):
        for axis, step in enumerate(o):
            if step:
                there = at[axis] + step
                inside[:, k] &= (there >= 0) & (there < dims[axis])
        cols[:, k] = (node + sum(s * step for s, step in zip(strides, o))).to(torch.int32)
    rowptr = torch.zeros(count + 1, dtype=torch.int32, device=DEVICE)
    rowptr[1:] = torch.cumsum(inside.sum(1), 0).to(torch.int32)
    vals = _uniform(g, count * len(offsets), -1.5, -0.5).reshape(count, len(offsets))
    centre = offsets.index((0,) * len(dims))
    vals[:, centre] = (len(offsets) - 1) - 0.5 * (1.0 + vals[:, centre])
    return count, count, rowptr, cols[inside], vals[inside]


def _random_rows(m, n, low, high, unsorted, pattern, g):
    """Rows of low..high entries at uniformly drawn columns (a column drawn twice is kept once)."""
    counts = torch.randint(low, high + 1, (m,), generator=pattern, device=DEVICE)
    rows = torch.repeat_interleave(torch.arange(m, device=DEVICE), counts)
    cols = torch.randint(0, n, (rows.numel(),), generator=pattern, device=DEVICE)
    keys = torch.unique(rows * n + cols)
    rowptr, colind = _from_keys(m, n, keys)
    if unsorted:
        rows = torch.div(keys, n, rounding_mode="floor")
        colind = colind[torch.argsort(rows + 0.999 * _uniform(pattern, keys.numel(), 0.0, 1.0))]
    return m, n, rowptr, colind, _uniform(g, keys.numel(), -1.0, 1.0)


def _rmat(scale, pattern, g):
    """R-MAT graph with 16 edges per vertex, repeated edges merged."""
    n = 1 << scale
    a, b, c = RMAT
    rows = torch.zeros(16 * n, dtype=torch.int64, device=DEVICE)
    cols = torch.zeros_like(rows)
    for _ in range(scale):
        u = torch.rand(16 * n, generator=pattern, device=DEVICE)
        rows = 2 * rows + (u >= a + b)
        cols = 2 * cols + (((u >= a) & (u < a + b)) | (u >= a + b + c))
    keys = torch.unique(rows * n + cols)
    rowptr, colind = _from_keys(n, n, keys)
    return n, n, rowptr, colind, _uniform(g, keys.numel(), -1.0, 1.0)


def _aggregates(dims):
    """Piecewise-constant prolongator over 2x2x2 node blocks, and its transpose."""
    coarse = [-(-d // 2) for d in dims]
    fine, nc = math.prod(dims), math.prod(coarse)
    node = torch.arange(fine, device=DEVICE)
    agg, stride, cstride = torch.zeros_like(node), 1, 1
    for d, c in zip(dims, coarse):
        agg += cstride * torch.div(torch.div(node, stride, rounding_mode="floor") % d, 2, rounding_mode="floor")
        stride *= d
        cstride *= c
    one = torch.ones(fine, dtype=torch.float64, device=DEVICE)
    P = (fine, nc, torch.arange(fine + 1, dtype=torch.int32, device=DEVICE), agg.to(torch.int32), one)
    rowptr = torch.zeros(nc + 1, dtype=torch.int32, device=DEVICE)
    rowptr[1:] = torch.cumsum(torch.bincount(agg, minlength=nc), 0).to(torch.int32)
    R = (nc, fine, rowptr, torch.argsort(agg, stable=True).to(torch.int32), one.clone())
    return P, R


def _batch_shapes(case):
    """Per pair of the batch: (grid dims, points of A, points of B), 0 points for random rows."""
    rng = np.random.RandomState(case["mix"])
    shapes = []
    for _ in range(case["count"]):
        r = math.exp(rng.uniform(math.log(case["rows_low"]), math.log(case["rows_high"])))
        nx = max(3, int(round(math.sqrt(r))))
        kinds = [int(rng.choice([0, 0, 5, 9])) for _ in range(2)]
        shapes.append(((nx, max(3, int(round(r / nx)))), *kinds))
    return shapes


def _operands(case, seed):
    """The case's matrices, as a list."""
    g = _generator(seed)
    pattern = _generator(case.get("pattern", case.get("mix", 0)))
    if case["op"] == "batch":
        mats = []
        for dims, *kinds in _batch_shapes(case):
            n = dims[0] * dims[1]
            mats += [_grid(dims, k, g) if k else _random_rows(n, n, 3, 40, False, pattern, g) for k in kinds]
        return mats
    if case["op"] in ("galerkin", "jacobi"):
        A = _grid(_dims(case), 7, g)
        P, R = _aggregates(_dims(case))
        return [A, P, R] if case["op"] == "galerkin" else [A, P]
    if case["op"] == "spadd":
        return [_random_rows(case["rows"], case["cols"], case["low"], case["high"], case["unsorted"], pattern, g)
                for _ in range(2)]
    if case["kind"] == "random":
        return [_random_rows(case["rows"], case["inner"], case["low"], case["high"], case["unsorted"], pattern, g),
                _random_rows(case["inner"], case["cols"], case["low"], case["high"], case["unsorted"], pattern, g)]
    A = _grid(_dims(case), case["points"], g) if case["kind"] == "grid" else _rmat(case["scale"], pattern, g)
    return [A, A]


def _samples(case, seed):
    """Row features, capacity classes and network parameters."""
    g = _generator(seed)
    X = _uniform(g, case["samples"] * K.MLP_FEATURES, 0.0, 18.0).reshape(-1, K.MLP_FEATURES).float()
    y = torch.randint(0, K.MLP_CLASSES, (case["samples"],), generator=g, device=DEVICE, dtype=torch.int32)
    params = []
    for rows, cols in ((8, 32), (32, 32), (32, 16)):
        params += [_uniform(g, rows * cols, -1.0, 1.0) * math.sqrt(6.0 / rows), _uniform(g, cols, -0.1, 0.1)]
    return X, y, torch.cat(params).float()


# ----------------------------------------------------------------------------
# One pass
# ----------------------------------------------------------------------------
def prepare(case, seed):
    op = case["op"]
    if op == "mlp_grad":
        X, y, params = _samples(case, seed)
        return {"op": op, "X": X, "y": y, "params": params, "grad": torch.empty_like(params),
                "loss": torch.empty(1, dtype=torch.float32, device=DEVICE)}
    made = {}
    mats = []
    for M in _operands(case, seed):
        if id(M) not in made:
            made[id(M)] = (K.DeviceCSR(*M), M)  # the tuple keeps its id taken
        mats.append(made[id(M)][0])
    state = {"op": op, "mats": mats}
    if op == "batch":
        state["handle"] = K.BatchedSpGEMM()
    elif op == "galerkin":
        state["handle"], state["second"] = K.SpGEMM(), K.SpGEMM()
    else:
        state["handle"] = K.SpGEMM(arith=case.get("arith", 0))
    if op == "refresh":
        rowptr, nnz = state["handle"].symbolic(*mats)
        colind = torch.empty(nnz, dtype=torch.int32, device=DEVICE)
        vals = torch.empty(nnz, dtype=torch.float64, device=DEVICE)
        state["c"] = (rowptr, nnz, colind, vals)
    for key in ("omega", "alpha", "beta"):
        if key in case:
            state[key] = case[key]
    return state


def run(state):
    op = state["op"]
    if op == "mlp_grad":
        K.kk_mlp_loss_grad(state["X"], state["y"], state["params"], state["grad"], state["loss"])
        return state["grad"], state["loss"]
    h, mats = state["handle"], state["mats"]
    if op == "product":
        rowptr, nnz = h.symbolic(*mats)
        return (rowptr, *h.numeric(*mats, rowptr, nnz))
    if op == "refresh":
        return h.numeric(*mats, *state["c"])
    if op == "learned":
        rowptr, nnz = h.learned_symbolic(*mats)
        return (rowptr, *h.learned_numeric(*mats, rowptr, nnz))
    if op == "jacobi":
        rowptr, nnz = h.symbolic(*mats)
        return (rowptr, *h.jacobi_numeric(*mats, rowptr, nnz, state["omega"]))
    if op == "spadd":
        rowptr, nnz = h.spadd_symbolic(*mats)
        return (rowptr, *h.spadd_numeric(state["alpha"], mats[0], state["beta"], mats[1], rowptr, nnz))
    if op == "batch":
        As, Bs = mats[0::2], mats[1::2]
        rowptr, offsets, total = h.symbolic(As, Bs)
        return (rowptr, offsets, *h.numeric(As, Bs, rowptr, total))
    A, P, R = mats
    rowptr, nnz = h.symbolic(A, P)
    colind, vals = h.numeric(A, P, rowptr, nnz)
    AP = K.DeviceCSR(A.m, P.n, rowptr.to(torch.int32), colind, vals)
    coarse, nnz = state["second"].symbolic(R, AP)
    return (rowptr, colind, vals, coarse, *state["second"].numeric(R, AP, coarse, nnz))


# ----------------------------------------------------------------------------
# What a pass cannot do without
# ----------------------------------------------------------------------------
def _grid_counts(dims, points):
    """(nnz of A, multiply-adds of A*A, nnz of A*A) of a grid operator."""
    reach = {}
    offsets = _offsets(points)
    for o in offsets:
        for p in offsets:
            reach[tuple(a + b for a, b in zip(o, p))] = True
    count = lambda o: math.prod(max(0, d - abs(s)) for d, s in zip(dims, o))  # noqa: E731
    # row length of every node, as a sum (5, 7 points) or a product over the axes
    axes = []
    for d in dims:
        near = np.full(d, 2)
        near[0] -= 1
        near[-1] -= 1
        axes.append(near)
    length = np.ones([1] * len(dims))
    for k, near in enumerate(axes):
        shape = [1] * len(dims)
        shape[k] = -1
        length = length + near.reshape(shape) if points in (5, 7) else length * (near + 1).reshape(shape)
    return sum(count(o) for o in offsets), float((length ** 2).sum()), sum(count(o) for o in reach)


def _distinct(n, drawn):
    return n * (1.0 - math.exp(-drawn / n))


def _random_counts(m, k, n, low, high):
    mid = 0.5 * (low + high)
    la, lb = _distinct(k, mid), _distinct(n, mid)
    return m * la, k * lb, m * la * lb, m * _distinct(n, la * lb)


def _csr_bytes(m, nnz):
    return 4.0 * (m + 1) + 12.0 * nnz


def _product_work(m, k, nnz_a, nnz_b, madds, nnz_c, same=False, refresh=False):
    inputs = _csr_bytes(m, nnz_a) + (0.0 if same else _csr_bytes(k, nnz_b))
    return {"bytes": inputs + 8.0 * (m + 1) + 12.0 * nnz_c, "flops": 2.0 * madds}


def _mixed_counts(dims, a, b):
    """(nnz of A, nnz of B, multiply-adds, nnz of C) of one pair of a batch."""
    n = dims[0] * dims[1]
    if a and a == b:
        nnz, madds, nnz_c = _grid_counts(dims, a)
        return nnz, nnz, madds, nnz_c
    if not a and not b:
        return _random_counts(n, n, n, 3, 40)
    nnz_a = _grid_counts(dims, a)[0] if a else n * _distinct(n, 21.5)
    nnz_b = _grid_counts(dims, b)[0] if b else n * _distinct(n, 21.5)
    madds = nnz_a * nnz_b / n
    return nnz_a, nnz_b, madds, min(madds, 25.0 * n) if a and b else n * _distinct(n, madds / n)


def work(case):
    op = case["op"]
    if op == "mlp_grad":
        # forward, and both products of backward (the first layer needs one)
        return {"bytes": case["samples"] * 36.0 + 2 * 1872 * 4.0, "flops": case["samples"] * 2.0 * (1792 * 3 - 256)}
    if op in ("galerkin", "jacobi"):
        dims = _dims(case)
        coarse = [-(-d // 2) for d in dims]
        m, mc = math.prod(dims), math.prod(coarse)
        nnz_a = _grid_counts(dims, 7)[0]
        # one further aggregate per axis, except at the ends of the grid
        nnz_ap = float(m + sum((d - 1 - (d % 2 == 0)) * (m // d) for d in dims))
        first = _product_work(m, m, nnz_a, m, nnz_a, nnz_ap)
        if op == "jacobi":
            return first
        second = _product_work(mc, m, m, nnz_ap, nnz_ap, _grid_counts(coarse, 7)[0])
        return {k: first[k] + second[k] for k in first}
    if op == "spadd":
        mid = _distinct(case["cols"], 0.5 * (case["low"] + case["high"]))
        m, nnz = case["rows"], case["rows"] * mid
        nnz_c = m * _distinct(case["cols"], 2 * mid)
        return {"bytes": 2 * _csr_bytes(m, nnz) + 8.0 * (m + 1) + 12.0 * nnz_c, "flops": 3.0 * nnz}
    if op == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for dims, a, b in _batch_shapes(case):
            n = dims[0] * dims[1]
            w = _product_work(n, n, *_mixed_counts(dims, a, b))
            total = {k: total[k] + w[k] for k in total}
        return total
    if case["kind"] == "grid":
        m = math.prod(_dims(case))
        nnz, madds, nnz_c = _grid_counts(_dims(case), case["points"])
        return _product_work(m, m, nnz, nnz, madds, nnz_c, same=True)
    if case["kind"] == "random":
        return _product_work(case["rows"], case["inner"], *_random_counts(
            case["rows"], case["inner"], case["cols"], case["low"], case["high"]), same=False)
    n = 1 << case["scale"]
    nnz, madds, nnz_c = (1e6 * v for v in RMAT_COUNTS[case["scale"]])
    return _product_work(n, n, nnz, nnz, madds, nnz_c, same=True)


# Scale: entries of the merged graph, multiply-adds of its square and entries of
# the square, in millions (means over three seeds, as counted).
RMAT_COUNTS = {
    10: (0.01215, 0.8138, 0.2673),
    11: (0.02563, 2.366, 0.8098),
    12: (0.05345, 6.747, 2.394),
    13: (0.1108, 19.04, 7.012),
    14: (0.2284, 53.22, 20.36),
    15: (0.4681, 146.5, 57.89),
    16: (0.9555, 400.1, 163.4),
    17: (1.943, 1086, 458.8),
    18: (3.94, 2929, 1277),
}


# ----------------------------------------------------------------------------
# The same results in plain 64-bit torch
# ----------------------------------------------------------------------------
def _sum_by_key(keys, vals):
    keys, order = torch.sort(keys, stable=True)
    found, back = torch.unique_consecutive(keys, return_inverse=True)
    return found, torch.zeros(found.numel(), dtype=torch.float64, device=DEVICE).index_add_(0, back, vals[order])


def _exact_product(A, B, most=1 << 27):
    """A*B by sorting all products of a block of rows at a time: rowptr (int64), colind, vals."""
    m, _, arp, acol, aval = A
    _, n, brp, bcol, bval = B
    arp, brp = arp.long(), brp.long()
    lengths = (brp[1:] - brp[:-1])[acol.long()]
    ends = torch.zeros(acol.numel() + 1, dtype=torch.int64, device=DEVICE)
    torch.cumsum(lengths, 0, out=ends[1:])
    row_ends = ends[arp]
    arows = torch.repeat_interleave(torch.arange(m, device=DEVICE), arp[1:] - arp[:-1])
    cols, vals, counts, r = [], [], torch.zeros(m, dtype=torch.int64, device=DEVICE), 0
    while r < m:
        stop = int(torch.searchsorted(row_ends, row_ends[r] + most, right=True)) - 1
        stop = min(m, max(r + 1, stop))
        p = slice(int(arp[r]), int(arp[stop]))
        entry = torch.repeat_interleave(torch.arange(p.start, p.stop, device=DEVICE), lengths[p])
        at = torch.arange(entry.numel(), device=DEVICE) + row_ends[r] - ends[entry] + brp[acol[entry].long()]
        keys, sums = _sum_by_key(arows[entry] * n + bcol[at], aval[entry] * bval[at])
        rows = torch.div(keys, n, rounding_mode="floor")
        counts += torch.bincount(rows, minlength=m)
        cols.append((keys - rows * n).to(torch.int32))
        vals.append(sums)
        r = stop
    rowptr = torch.zeros(m + 1, dtype=torch.int64, device=DEVICE)
    torch.cumsum(counts, 0, out=rowptr[1:])
    return rowptr, torch.cat(cols), torch.cat(vals)


def _rows_of(M):
    return torch.repeat_interleave(torch.arange(M[0], device=DEVICE), (M[2][1:] - M[2][:-1]).long())


def _exact_gradient(case, seed):
    X, y, params = _samples(case, seed)
    X, theta = X.double(), params.double().requires_grad_()
    parts = torch.split(theta, [256, 32, 1024, 32, 512, 16])
    h = torch.relu(X @ parts[0].reshape(8, 32) + parts[1])
    h = torch.relu(h @ parts[2].reshape(32, 32) + parts[3])
    loss = torch.nn.functional.cross_entropy(h @ parts[4].reshape(32, 16) + parts[5], y.long())
    loss.backward()
    return theta.grad, loss.detach().reshape(1)


def exact(case, seed):
    op = case["op"]
    if op == "mlp_grad":
        return _exact_gradient(case, seed)
    mats = _operands(case, seed)
    if op == "spadd":
        A, B = mats
        n = A[1]
        keys = torch.cat([_rows_of(M) * n + M[3] for M in mats])
        found, sums = _sum_by_key(keys, torch.cat([case["alpha"] * A[4], case["beta"] * B[4]]))
        rowptr, colind = _from_keys(A[0], n, found)
        return rowptr.long(), colind, sums
    if op == "batch":
        parts = [_exact_product(A, B) for A, B in zip(mats[0::2], mats[1::2])]
        ends = np.cumsum([0] + [p[1].numel() for p in parts])
        rowptr = torch.cat([p[0][:-1] + int(e) for p, e in zip(parts, ends)])
        rowptr = torch.cat([rowptr, rowptr.new_tensor([int(ends[-1])])])
        return rowptr, ends.astype(np.int64), torch.cat([p[1] for p in parts]), torch.cat([p[2] for p in parts])
    if op == "jacobi":
        A, P = mats
        on = A[3] == _rows_of(A)  # every row has one diagonal entry, in row order
        diagonal = A[4][on]
        scaled = -case["omega"] / diagonal[_rows_of(A)] * A[4]
        scaled[on] += 1.0
        return _exact_product((*A[:4], scaled), P)
    if op == "galerkin":
        A, P, R = mats
        first = _exact_product(A, P)
        return (*first, *_exact_product(R, (A[0], P[1], *first)))
    rowptr, colind, vals = _exact_product(*mats)
    return (colind, vals) if op == "refresh" else (rowptr, colind, vals)
