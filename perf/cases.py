"""Performance cases: the work a program hands to this library, through its public entry points.

Every case is one call pattern on one 0-1 ILP:

- ``iterate``: a solver is in hand; a pass runs ``iters`` iterations on the device and returns the
  bound after each of them, the multipliers and (``mm``) the min-marginals;
- ``resolve``: a solver is in hand; a pass gives it new costs from the host, iterates, and reads
  bound, multipliers and min-marginals back to host arrays (the same model solved again and again);
- ``solve``: a pass builds the solver from host arrays, iterates, reads everything back and frees it;
- ``smooth``: a pass is a training step's share of this library: the smoothed bound of ``iters``
  iterations and its gradient in the costs.

Families and sizes are those of the workloads of this repository (Potts MRF, sparse matching,
discrete tomography, cell tracking, batches of uneven Potts grids) and of its tests (rows of several
hundred variables), down to the smallest calls.
"""
from __future__ import annotations

from types import SimpleNamespace

import numpy as np
import torch

OMEGA = 0.5


# ------------------------------------------------------------------------------------------
# cases
# ------------------------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: one iteration on a toy grid, as a solver stepped from a host loop does
        # between its own checks (launches and latency only)
        dict(name="step_potts_6x6x3", use="iterate", family="potts", H=6, W=6, L=3, iters=1, mm=False),
        # one small MRF, the 20x20x3 workload with its 100 iterations
        dict(name="potts_20x20x3", use="iterate", family="potts", H=20, W=20, L=3, iters=100, mm=True),
        # the 300x300 matching workload: many two-variable rows, variables in some fifteen rows
        dict(name="matching_300", use="iterate", family="matching", left=300, right=300, k=10, pairs=20000,
             iters=100, mm=True),
        # the 64x64x3 tomography workload: long wide projection rows beside a Potts grid
        dict(name="tomography_64", use="iterate", family="tomography", side=64, levels=3, iters=100, mm=True),
        # the 50x200 cell-tracking workload with its 50 iterations: rows of 15 to 30 variables
        dict(name="tracking_50x200", use="iterate", family="tracking", frames=50, dets=200, knn=5, iters=50, mm=True),
        # many uneven Potts grids (sides 16..128, labels 2..8) packed into one solver: throughput
        dict(name="batch_32", use="iterate", family="batch", count=32, iters=20, mm=True),
        # rows of up to 300 variables, BDD layers up to 150 nodes wide
        dict(name="wide_rows_300", use="iterate", family="wide", n=2000, rows=300, longest=300, iters=50, mm=True),
        # the tomography workload with its long rows cut into pieces of at most 32 layers
        dict(name="split_tomography_64", use="iterate", family="tomography", side=64, levels=3, split=32, iters=100,
             mm=True),
        # the matching model solved again with new costs from the host, a short solve
        dict(name="resolve_matching_300", use="resolve", family="matching", left=300, right=300, k=10, pairs=20000,
             iters=20),
        # one model solved from scratch: compile, upload, iterate, read back
        dict(name="solve_potts_64x64x4", use="solve", family="potts", H=64, W=64, L=4, iters=100),
        # learning costs on the tracking workload: smoothed bound of 50 iterations and its gradient
        dict(name="smooth_tracking_50x200", use="smooth", family="tracking", frames=50, dets=200, knn=5, iters=50,
             alpha=0.1),
        # the same on tomography, whose projection rows are wide
        dict(name="smooth_tomography_32", use="smooth", family="tomography", side=32, levels=3, iters=20, alpha=0.1),
    ]


def draw(rng):
    """One more case: any family, sizes spread over the logarithm of the listed ranges."""
    def log(a, b):
        return int(round(a * (b / a) ** rng.random()))

    kind = rng.choice(["potts", "matching", "tomography", "tracking", "batch", "wide", "split", "resolve", "solve",
                       "smooth_tracking", "smooth_tomography"])
    iters = log(1, 100)
    if kind == "potts":
        return dict(use="iterate", family="potts", H=log(4, 96), W=log(4, 96), L=rng.randint(2, 8), iters=iters,
                    mm=rng.random() < 0.7)
    if kind in ("matching", "resolve"):
        left = log(20, 300)
        right = max(12, int(left * rng.uniform(0.7, 1.3)))
        k = rng.randint(3, 10)
        most = min(60 * left, (left * k) ** 2 // 8)  # far below the number of distinct pairs
        case = dict(use="iterate", family="matching", left=left, right=right, k=k,
                    pairs=log(min(5 * left, most), most), iters=iters, mm=True)
        if kind == "resolve":
            case.update(use="resolve", iters=log(5, 50))
            del case["mm"]
        return case
    if kind in ("tomography", "split"):
        case = dict(use="iterate", family="tomography", side=log(8, 64), levels=rng.randint(2, 3), iters=iters, mm=True)
        if kind == "split":
            case["split"] = log(8, 64)
        return case
    if kind == "tracking":
        return dict(use="iterate", family="tracking", frames=log(3, 50), dets=log(10, 200), knn=rng.randint(3, 5),
                    iters=min(iters, 50), mm=True)
    if kind == "batch":
        return dict(use="iterate", family="batch", count=log(2, 32), iters=min(iters, 20), mm=rng.random() < 0.7)
    if kind == "wide":
        return dict(use="iterate", family="wide", n=log(300, 4000), rows=log(20, 300), longest=log(40, 300),
                    iters=min(iters, 50), mm=True)
    if kind == "solve":
        return dict(use="solve", family="potts", H=log(8, 64), W=log(8, 64), L=rng.randint(2, 6), iters=iters)
    if kind == "smooth_tracking":
        return dict(use="smooth", family="tracking", frames=log(3, 50), dets=log(10, 200), knn=rng.randint(3, 5),
                    iters=min(iters, 50), alpha=rng.choice([0.1, 0.2, 0.5]))
    return dict(use="smooth", family="tomography", side=log(8, 32), levels=3, iters=min(iters, 20),
                alpha=rng.choice([0.1, 0.2, 0.5]))


# ------------------------------------------------------------------------------------------
# instances: integer constraint matrices in CSR form and costs, from a seed alone
# ------------------------------------------------------------------------------------------

def _assemble(n, lens, col, val, b, sense, c):
    row_ptr = np.zeros(len(lens) + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    return SimpleNamespace(n=int(n), m=len(lens), nnz=int(row_ptr[-1]), row_ptr=row_ptr,
                           col=np.ascontiguousarray(col, np.int32), val=np.ascontiguousarray(val, np.int32),
                           b=np.ascontiguousarray(b, np.int32), sense=np.ascontiguousarray(sense, np.int8),
                           c=np.ascontiguousarray(c, np.float32))


def _grid(H, W, L, unary, weight):
    """Local-polytope ILP of a 4-connected Potts grid: sum_l x_il = 1 per pixel; per edge and label
    sum_l' y_ll' = x_il and sum_l y_ll' = x_jl'.  (n, row lengths, columns, values, b, costs)"""
    p = np.arange(H * W, dtype=np.int64).reshape(H, W)
    src = np.concatenate([p[:, :-1].ravel(), p[:-1, :].ravel()])
    dst = np.concatenate([p[:, 1:].ravel(), p[1:, :].ravel()])
    order = np.argsort(src, kind="stable")
    src, dst = src[order], dst[order]
    E, nx, lab = len(src), H * W * L, np.arange(L, dtype=np.int64)
    y = nx + (np.arange(E)[:, None, None] * L + lab[:, None]) * L + lab
    col = np.empty((E, 2, L, L + 1), np.int64)
    col[:, 0, :, 0] = src[:, None] * L + lab
    col[:, 1, :, 0] = dst[:, None] * L + lab
    col[:, 0, :, 1:] = y
    col[:, 1, :, 1:] = y.transpose(0, 2, 1)
    val = np.ones((E * 2 * L, L + 1), np.int32)
    val[:, 0] = -1
    lens = np.concatenate([np.full(H * W, L), np.full(E * 2 * L, L + 1)])
    b = np.concatenate([np.ones(H * W, np.int32), np.zeros(E * 2 * L, np.int32)])
    pair = (weight * (lab[:, None] != lab)).astype(np.float32).ravel()
    return (nx + E * L * L, lens, np.concatenate([np.arange(nx), col.ravel()]),
            np.concatenate([np.ones(nx, np.int32), val.ravel()]), b,
            np.concatenate([unary.ravel().astype(np.float32), np.tile(pair, E)]))


def _potts(shapes, rng):
    """Independent Potts grids (H, W, L), one after another."""
    parts, off = [], 0
    for H, W, L in shapes:
        n, lens, col, val, b, c = _grid(H, W, L, rng.standard_normal(H * W * L), 0.5)
        parts.append((lens, col + off, val, b, c))
        off += n
    lens, col, val, b, c = (np.concatenate(x) for x in zip(*parts))
    return _assemble(off, lens, col, val, b, np.zeros(len(b)), c)


def _matching(left, right, k, pairs, rng):
    """Sparse graph matching: k candidates per left point, sum = 1 per left and <= 1 per right point,
    quadratic pairs z <= x, z <= x'."""
    k = min(k, right)
    cand = np.sort(np.argsort(rng.random((left, right)), axis=1)[:, :k], axis=1)
    nx, xl, xr = left * k, np.repeat(np.arange(left), k), cand.ravel()
    by_right = np.argsort(xr, kind="stable")
    counts = np.bincount(xr, minlength=right)
    counts = counts[counts > 0]
    a, z = rng.integers(0, nx, 6 * pairs), rng.integers(0, nx, 6 * pairs)
    lo, hi = np.minimum(a, z), np.maximum(a, z)
    ok = (xl[lo] != xl[hi]) & (xr[lo] != xr[hi])
    _, first = np.unique(lo[ok] * nx + hi[ok], return_index=True)
    first = np.sort(first)[:pairs]
    lo, hi = lo[ok][first], hi[ok][first]
    np_ = len(lo)
    zid = nx + np.arange(np_)
    pcol = np.stack([lo, zid, hi, zid], axis=1).ravel()
    lens = np.concatenate([np.full(left, k), counts, np.full(2 * np_, 2)])
    col = np.concatenate([np.arange(nx), by_right, pcol])
    val = np.concatenate([np.ones(2 * nx, np.int32), np.tile(np.array([-1, 1], np.int32), 2 * np_)])
    b = np.concatenate([np.ones(left + len(counts), np.int32), np.zeros(2 * np_, np.int32)])
    sense = np.concatenate([np.zeros(left), np.full(len(counts) + 2 * np_, -1)])
    c = np.concatenate([rng.uniform(-1, 0, nx), rng.normal(0, 0.3, np_)])
    return _assemble(nx + np_, lens, col, val, b, sense, c)


def _tomography(side, levels, rng):
    """Potts grid (weight 0.2, small unaries) plus projection equalities sum_l l x = p along rows,
    columns and both diagonals of a piecewise-constant image."""
    pts, lev = rng.uniform(0, side, (16, 2)), rng.integers(0, levels, 16)
    rr, cc = np.meshgrid(np.arange(side) + 0.5, np.arange(side) + 0.5, indexing="ij")
    img = lev[np.argmin((rr[..., None] - pts[:, 0]) ** 2 + (cc[..., None] - pts[:, 1]) ** 2, axis=-1)].ravel()
    n, lens, col, val, b, c = _grid(side, side, levels, rng.normal(0, 0.01, side * side * levels), 0.2)
    idx = np.arange(side * side).reshape(side, side)
    lines = [idx[r] for r in range(side)] + [idx[:, r] for r in range(side)]
    for g in (idx, idx[:, ::-1]):
        lines += [np.sort(np.diagonal(g, offset=o)) for o in range(-(side - 1), side)]
    steps = np.arange(1, levels)
    pcol = [(ln[:, None] * levels + steps).ravel() for ln in lines]
    pval = [np.tile(steps, len(ln)) for ln in lines]
    pb = [int(img[ln].sum()) for ln in lines]
    lens = np.concatenate([lens, [len(x) for x in pcol]])
    b = np.concatenate([b, pb])
    return _assemble(n, lens, np.concatenate([col] + pcol), np.concatenate([val] + pval), b, np.zeros(len(b)), c)


def _tracking(frames, dets, knn, rng):
    """Cell tracking as a flow: appear, disappear and detection variables, transitions to the knn
    nearest detections of the next frame, divisions into pairs of them."""
    knn = min(knn, dets)
    pos = rng.uniform(0, 1, (frames, dets, 2))
    D, S = frames * dets, (frames - 1) * dets
    first, second = np.triu_indices(knn, 1)
    q = len(first)
    t0 = 3 * D
    d0 = t0 + S * knn
    n = d0 + S * q
    d2 = ((pos[:-1, :, None] - pos[1:, None]) ** 2).sum(-1)
    nn = np.sort(np.argpartition(d2, knn - 1, axis=2)[:, :, :knn], axis=2).reshape(S, knn)
    nbr = nn + np.repeat(np.arange(1, frames), dets)[:, None] * dets
    tid = t0 + np.arange(S * knn).reshape(S, knn)
    did = d0 + np.arange(S * q).reshape(S, q)
    det = np.arange(D)
    # entries (row, column, value): in-flow rows, out-flow rows, children rows
    rows = [det, det, nbr.ravel(), nbr[:, first].ravel(), nbr[:, second].ravel(), D + det, D + det]
    cols = [3 * det, 3 * det + 1, tid.ravel(), did.ravel(), did.ravel(), 3 * det, 3 * det + 2]
    vals = [-1, 1, 1, 1, 1, -1, 1]
    src = np.arange(S)
    for base, v in ((D, 1), (2 * D, 2)):
        rows += [np.repeat(base + src, knn), np.repeat(base + src, q)]
        cols += [tid.ravel(), did.ravel()]
        vals += [1, v]
    val = np.concatenate([np.full(len(r), v) for r, v in zip(rows, vals)])
    row, col = np.concatenate(rows), np.concatenate(cols)
    order = np.lexsort((col, row))
    m = 2 * D + S
    lens = np.bincount(row, minlength=m)
    b = np.concatenate([np.zeros(2 * D), np.full(S, 2)])
    sense = np.concatenate([np.zeros(2 * D), np.full(S, -1)])
    return _assemble(n, lens, col[order], val[order], b, sense, rng.standard_normal(n))


def _wide_lengths(n, rows, longest):
    """Row lengths of a `wide` case: 4 to `longest`, spread over their logarithm."""
    longest = min(longest, n)
    return np.round(4 * (longest / 4) ** np.linspace(0, 1, rows)).astype(np.int64)[::-1]


def _wide(n, rows, longest, rng):
    """At-most-half rows over 4 to `longest` of n variables."""
    lens = rng.permutation(_wide_lengths(n, rows, longest))
    col = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens])
    return _assemble(n, lens, col, np.ones(len(col)), lens // 2, np.full(rows, -1), rng.standard_normal(n))


def _batch_shapes(count, rng):
    return [(s, s, int(rng.integers(2, 9))) for s in rng.integers(16, 129, count).tolist()]


def _instance(case, seed):
    rng = np.random.default_rng([seed, 77])
    f = case["family"]
    if f == "potts":
        return _potts([(case["H"], case["W"], case["L"])], rng)
    if f == "batch":
        # the shapes are the case's, the costs the seed's: every pass moves the same bytes
        return _potts(_batch_shapes(case["count"], np.random.default_rng(case["count"])), rng)
    if f == "matching":
        return _matching(case["left"], case["right"], case["k"], case["pairs"], rng)
    if f == "tomography":
        return _tomography(case["side"], case["levels"], rng)
    if f == "tracking":
        return _tracking(case["frames"], case["dets"], case["knn"], rng)
    return _wide(case["n"], case["rows"], case["longest"], rng)


# ------------------------------------------------------------------------------------------
# what is measured
# ------------------------------------------------------------------------------------------

def prepare(case, seed):
    from paper_2009_00481_gb300 import Solver
    inst = _instance(case, seed)
    use = case["use"]
    state = SimpleNamespace(case=case, inst=inst)
    if use == "solve":
        return state
    state.solver = Solver(inst, omega=OMEGA, alpha=case.get("alpha", 0.0), split_depth=case.get("split", 0))
    dev = torch.device("cuda", torch.cuda.current_device())
    if use == "iterate":
        state.trace = torch.empty(case["iters"], dtype=torch.float64, device=dev)
        state.lam = torch.empty(inst.nnz, dtype=torch.float32, device=dev)
        state.mm = [torch.empty(inst.nnz, dtype=torch.float32, device=dev) for _ in range(2)] if case["mm"] else None
    elif use == "resolve":
        state.costs = _fresh_costs(inst, seed)
    else:
        state.c = torch.from_numpy(inst.c).to(dev).requires_grad_(True)
    return state


def _fresh_costs(inst, seed):
    scale = 1.0 + 0.2 * np.random.default_rng([seed, 78]).standard_normal(inst.n)
    return (inst.c * scale).astype(np.float32)


def run(state):
    case, use = state.case, state.case["use"]
    if use == "iterate":
        m0, m1 = state.mm or (None, None)
        state.solver.iterate_device(case["iters"], trace=state.trace, lam=state.lam, mm0=m0, mm1=m1)
        out = {"trace": state.trace, "lam": state.lam}
        return dict(out, mm0=m0, mm1=m1) if state.mm else out
    if use == "smooth":
        from paper_2009_00481_gb300 import smoothed_bound
        state.c.grad = None
        bound = smoothed_bound(state.c, state.solver, case["iters"])
        bound.backward()
        return {"bound": bound.detach(), "grad": state.c.grad}
    if use == "resolve":
        state.solver.set_costs(state.costs)
        bound, lam, m0, m1 = state.solver.iterate(case["iters"], lam=True, mm=True)
    else:
        from paper_2009_00481_gb300 import Solver
        solver = Solver(state.inst, omega=OMEGA)
        bound, lam, m0, m1 = solver.iterate(case["iters"], lam=True, mm=True)
        solver.close()
    return {"bound": bound, "lam": lam, "mm0": m0, "mm1": m1}


def _sizes(case):
    """(variables, rows, nonzeros, BDD nodes) of a case, the nodes from each row's widest layer."""
    f = case["family"]
    if f in ("potts", "batch"):
        shapes = [(case["H"], case["W"], case["L"])] if f == "potts" else \
            _batch_shapes(case["count"], np.random.default_rng(case["count"]))
        n = m = nnz = 0
        for H, W, L in shapes:
            E = H * (W - 1) + W * (H - 1)
            n += H * W * L + E * L * L
            m += H * W + 2 * E * L
            nnz += H * W * L + 2 * E * L * (L + 1)
        return n, m, nnz, 2 * nnz - m
    if f == "matching":
        nx, p = case["left"] * case["k"], case["pairs"]
        return nx + p, case["left"] + case["right"] + 2 * p, 2 * nx + 4 * p, 4 * nx + 6 * p
    if f == "tomography":
        s, L = case["side"], case["levels"]
        E, px = 2 * s * (s - 1), s * s
        line = 4 * px * (L - 1)
        nnz = px * L + 2 * E * L * (L + 1) + line
        return (px * L + E * L * L, px + 2 * E * L + 6 * s - 2, nnz,
                2 * nnz + line * min(s, 40) * (L - 1) // 2)
    if f == "tracking":
        S, q = (case["frames"] - 1) * case["dets"], case["knn"] * (case["knn"] - 1) // 2
        D = case["frames"] * case["dets"]
        nnz = 4 * D + S * (3 * case["knn"] + 4 * q)
        return 3 * D + S * (case["knn"] + q), 2 * D + S, nnz, 2 * nnz
    lens = _wide_lengths(case["n"], case["rows"], case["longest"])
    return case["n"], case["rows"], int(lens.sum()), int((lens * lens // 4).sum())


def work(case):
    """One pass cannot do without: the constraint matrix and costs read once (column, value), every
    output written once, and in each of an iteration's two sweeps every multiplier read and
    written and every node's two arcs relaxed in each direction (an addition and a minimum each) and
    added up into the min-marginals.  A smoothed step walks every sweep twice and keeps each sweep's
    multipliers for the way back."""
    n, m, nnz, nodes = _sizes(case)
    iters, use = case["iters"], case["use"]
    outputs = {"iterate": 4 * nnz * (3 if case.get("mm") else 1) + 8 * iters, "smooth": 4 * n + 8}
    moved = 8 * nnz + 4 * n + 5 * m + outputs.get(use, 12 * nnz + 8)
    sweeps = 2 * iters
    if use == "smooth":
        return {"bytes": moved + sweeps * nnz * 16, "flops": sweeps * nodes * 40}
    return {"bytes": moved + sweeps * nnz * 8, "flops": sweeps * nodes * 12}


# ------------------------------------------------------------------------------------------
# 64-bit reference: the same schedule on partial sums instead of decision diagrams
# ------------------------------------------------------------------------------------------
# A row's messages live on its partial coefficient sums (the diagram merges sums that behave
# alike, which changes no path and so no message at a sum).  Infeasible states hold BIG.

BIG = 1e12
FORCED = 1e11


class _Rows:
    """Rows of about the same length, padded to one depth: [rows, depth] positions and values."""

    def __init__(self, inst, rows, depth, dev):
        ptr = inst.row_ptr[rows]
        lens = inst.row_ptr[rows + 1] - ptr
        k = np.arange(depth)
        act = k < lens[:, None]
        pos = np.where(act, ptr[:, None] + k, 0)
        a = np.where(act, inst.val[pos], 0)
        low = np.minimum(a, 0).sum(1)
        self.S = int((np.maximum(a, 0).sum(1) - low).max()) + 1
        self.depth, self.dev = depth, dev
        s = np.arange(self.S) + low[:, None]
        b, sense = inst.b[rows][:, None], inst.sense[rows][:, None]
        ok = np.where(sense == 0, s == b, np.where(sense < 0, s <= b, s >= b))
        self.final = torch.from_numpy(np.where(ok, 0.0, BIG)).to(dev)
        start = np.full((len(rows), self.S), BIG)
        start[np.arange(len(rows)), -low] = 0.0
        self.start = torch.from_numpy(start).to(dev)
        self.root = torch.from_numpy(-low).to(dev)[:, None]
        self.pos = torch.from_numpy(pos).to(dev)
        self.act = torch.from_numpy(act).to(dev)
        self.shift = [self._index(a[:, l], d) for l in range(depth) for d in (1, -1)]
        self.flat = torch.from_numpy(pos[act]).to(dev)

    def _index(self, a, sign):
        if (a == a[0]).all():
            return int(sign * a[0])
        i = np.arange(self.S) + sign * a[:, None]
        bad = (i < 0) | (i >= self.S)
        return torch.from_numpy(np.where(bad, 0, i)).to(self.dev), torch.from_numpy(bad).to(self.dev)

    def moved(self, x, l, sign):
        """x at the sums that the 1-arc of layer l leads to (sign 1) or comes from (sign -1)."""
        t = self.shift[2 * l + (0 if sign > 0 else 1)]
        if isinstance(t, int):
            pad = x.new_full((x.shape[0], min(abs(t), self.S)), BIG)
            if t == 0:
                return x
            return torch.cat([x[:, t:], pad], 1) if t > 0 else torch.cat([pad, x[:, :t]], 1)
        return torch.gather(x, 1, t[0]).masked_fill(t[1], BIG)


class _Exact:
    def __init__(self, inst, alpha):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.alpha, self.inst = alpha, inst
        lens = np.diff(inst.row_ptr)
        up = np.where(lens <= 10, lens, np.where(lens <= 32, -(-lens // 8) * 8, -(-lens // 32) * 32))
        self.groups = [_Rows(inst, np.nonzero(up == d)[0], int(d), self.dev) for d in np.unique(up)]
        self.back = torch.argsort(torch.cat([g.flat for g in self.groups]))
        self.var = torch.from_numpy(inst.col.astype(np.int64)).to(self.dev)
        self.deg = torch.bincount(self.var, minlength=inst.n).double()

    def least(self, a, b):
        if not self.alpha:
            return torch.minimum(a, b)
        return -self.alpha * torch.logaddexp(-a / self.alpha, -b / self.alpha)

    def least_of(self, x):
        if not self.alpha:
            return x.min(1).values
        return -self.alpha * torch.logsumexp(-x / self.alpha, 1)

    def one(self, g, l, lam, x):
        """x + lam where layer l of the row exists: the 1-arc's cost."""
        return torch.where(g.act[:, l:l + 1], x + lam[:, None], BIG)

    def backward_messages(self, g, lam):
        B = [g.final]
        for l in range(g.depth - 1, -1, -1):
            B.append(self.least(B[-1], self.one(g, l, lam[:, l], g.moved(B[-1], l, 1))))
        return B[::-1]

    def forward_messages(self, g, lam):
        F = [g.start]
        for l in range(g.depth):
            F.append(self.least(F[-1], self.one(g, l, lam[:, l], g.moved(F[-1], l, -1))))
        return F

    def marginals(self, g, l, lam, F, Bn):
        return self.least_of(F + Bn), self.least_of(self.one(g, l, lam, F + g.moved(Bn, l, 1)))

    def sweep(self, lam, share, msgs, forward):
        """One sweep over every row: (multipliers, differences, messages it leaves behind)."""
        lams, diffs, left = [], [], []
        for g, M in zip(self.groups, msgs):
            old = lam[g.pos] + share[g.pos]
            X = [g.start] if forward else [g.final]
            new, dif = [None] * g.depth, [None] * g.depth
            for l in (range(g.depth) if forward else range(g.depth - 1, -1, -1)):
                F, Bn = (X[-1], M[l + 1]) if forward else (M[l], X[-1])
                m0, m1 = self.marginals(g, l, old[:, l], F, Bn)
                free = (m0 < FORCED) & (m1 < FORCED) & g.act[:, l]
                d = OMEGA * torch.where(free, m1 - m0, torch.zeros_like(m0))
                new[l], dif[l] = old[:, l] - d, d
                X.append(self.least(X[-1], self.one(g, l, new[l], g.moved(X[-1], l, -1 if forward else 1))))
            left.append(X if forward else X[::-1])
            lams.append(torch.stack(new, 1)[g.act])
            diffs.append(torch.stack(dif, 1)[g.act])
        return torch.cat(lams)[self.back], torch.cat(diffs)[self.back], left

    def pending(self, diff):
        P = torch.zeros(self.inst.n, dtype=torch.float64, device=self.dev).index_add(0, self.var, diff)
        return P, (P / self.deg.clamp(min=1))[self.var]

    def slack(self, P):
        zero = torch.zeros_like(P)
        return self.least(P, zero) if self.alpha else torch.minimum(P, zero)

    def solve(self, c, iters):
        """Bounds after every iteration, multipliers with the pending share folded in."""
        lam = (c / self.deg.clamp(min=1))[self.var]
        share = torch.zeros_like(lam)
        msgs = [self.backward_messages(g, lam[g.pos]) for g in self.groups]
        trace = []
        empty = self.deg == 0
        for _ in range(iters):
            lam, diff, msgs = self.sweep(lam, share, msgs, True)
            _, share = self.pending(diff)
            lam, diff, msgs = self.sweep(lam, share, msgs, False)
            P, share = self.pending(diff)
            energy = sum(torch.gather(M[0], 1, g.root).sum() for g, M in zip(self.groups, msgs))
            trace.append(energy + self.slack(torch.where(empty, c, P)).sum())
        return torch.stack(trace), lam + share

    def min_marginals(self, lam):
        out = []
        for g in self.groups:
            x = lam[g.pos]
            F, B = self.forward_messages(g, x), self.backward_messages(g, x)
            both = [self.marginals(g, l, x[:, l], F[l], B[l + 1]) for l in range(g.depth)]
            out.append([torch.stack([m[k] for m in both], 1)[g.act] for k in (0, 1)])
        res = [torch.cat([o[k] for o in out])[self.back] for k in (0, 1)]
        return [torch.where(r < FORCED, r, torch.inf) for r in res]


def exact(case, seed):
    if case.get("split"):  # copy-arc duals belong to the reduced diagrams' arcs, not to the partial sums
        return None
    inst = _instance(case, seed)
    ref = _Exact(inst, case.get("alpha", 0.0))
    costs = _fresh_costs(inst, seed) if case["use"] == "resolve" else inst.c
    c = torch.from_numpy(costs).to(ref.dev).double()
    if case["use"] == "smooth":
        c.requires_grad_(True)
        trace, _ = ref.solve(c, case["iters"])
        trace[-1].backward()
        return {"bound": trace[-1].detach(), "grad": c.grad}
    with torch.no_grad():
        trace, lam = ref.solve(c, case["iters"])
        if case["use"] == "iterate":
            out = {"trace": trace, "lam": lam}
            return dict(out, **dict(zip(("mm0", "mm1"), ref.min_marginals(lam)))) if case["mm"] else out
        m0, m1 = ref.min_marginals(lam)
        return {"bound": trace[-1], "lam": lam, "mm0": m0, "mm1": m1}
