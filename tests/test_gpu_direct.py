"""The direct plan (plain solvers with default options: sweeps that form the pending shares themselves,
no pending passes between them) against the general plan, which an explicit layout option selects.
Both run the same operations on the same values, so multipliers, pending sums and min-marginals are
bit-identical and the bounds differ at most in the order of their FP64 sums (1e-12).  The cases sit
at the edges of the forms an instance can take: variables in 1, 2, 3..8, 9..16, 17..32 and more rows
(each its own way to a share), tiles of every register depth and the deep ones, chain and other layers,
layers of up to four nodes, tiles of mixed depth, rows with zero coefficients and variables in no row."""
from __future__ import annotations

import numpy as np
import pytest

from instances import SENSE_EQ, SENSE_GE, SENSE_LE, potts_batch, sparse_matching
from instances.generators import _from_rows

pytestmark = pytest.mark.gpu

ITERS = 19  # graphs of 8 iterations and a ragged tail


def rows_of(kind, cols):
    """One row over `cols`: at most one, exactly one, a flow row, at least one; layers of three and four
    nodes: children (some count twice, at most two), at most / exactly three."""
    ones = np.ones(len(cols), np.int64)
    if kind == "children":
        return (cols, 1 + (np.arange(len(cols)) >= len(cols) // 3), 2, SENSE_LE)
    if kind in ("three", "exactly_three"):
        return (cols, ones, 3, SENSE_LE if kind == "three" else SENSE_EQ)
    if kind == "flow":
        return (cols, np.concatenate([[-1], ones[1:]]), 0, SENSE_EQ)
    return (cols, ones, 1, {"most": SENSE_LE, "one": SENSE_EQ, "least": SENSE_GE}[kind])


def instance(degree, depths, kinds, rows_per_depth=40, seed=0):
    """Rows of the given depths over variables that lie in about `degree` rows each."""
    rng = np.random.default_rng([seed, degree])
    sizes = np.repeat(depths, rows_per_depth)
    n = max(int(np.ceil(sizes.sum() / degree)), int(max(depths)))
    rows = []
    left = np.full(n, degree)
    for k, d in enumerate(sizes):
        order = rng.permutation(n)
        cols = np.sort(order[np.argsort(-left[order], kind="stable")][:d])  # the fullest first: even degrees
        left[cols] -= 1
        rows.append(rows_of(kinds[k % len(kinds)], cols))
    return _from_rows(f"degree_{degree}", n + 3, rows, rng.standard_normal(n + 3).astype(np.float32))


def solver(inst, **kw):
    from paper_2009_00481_gb300 import Solver
    return Solver(inst, **kw)


def trace(s, iters=ITERS):
    import torch
    t = torch.zeros(iters, dtype=torch.float64, device="cuda")
    s.iterate_device(iters, trace=t)
    torch.cuda.synchronize()
    return t.cpu().numpy()


def close(a, b):
    a, b = np.asarray(a), np.asarray(b)
    assert np.all(np.abs(a - b) <= 1e-12 * np.maximum(1.0, np.abs(b))), np.abs(a - b).max()


def same(inst, **kw):
    a, b = solver(inst, **kw), solver(inst, lanes=0, tune_layout=0, staging=0, **kw)
    close(trace(a), trace(b))
    la, pa = a.get_state()
    lb, pb = b.get_state()
    np.testing.assert_array_equal(la, lb)
    np.testing.assert_array_equal(pa, pb)
    oa, ob = a.iterate(0, lam=True, mm=True), b.iterate(0, lam=True, mm=True)
    close(oa[0], ob[0])
    for x, y in zip(oa[1:], ob[1:]):
        np.testing.assert_array_equal(x, y)
    # from a state that is set (pending sums in the first row's difference), one iteration at a time
    c, d = solver(inst, **kw), solver(inst, lanes=0, tune_layout=0, staging=0, **kw)
    c.set_state(la, pa)
    d.set_state(la, pa)
    for _ in range(3):
        close(trace(c, 1), trace(d, 1))
    np.testing.assert_array_equal(c.get_state()[0], d.get_state()[0])
    parts = np.array([0, inst.m]), np.array([0, inst.n])
    close(a.bound_parts(*parts), b.bound_parts(*parts))
    # new costs restart both
    costs = (inst.c * 0.5 + 0.25).astype(np.float32)
    a.set_costs(costs)
    b.set_costs(costs)
    close(trace(a, 9), trace(b, 9))
    return a


@pytest.mark.parametrize("degree", [1, 2, 3, 4, 5, 8, 9, 16, 17, 32, 33, 70])
def test_variable_degrees(cuda_lib, degree):
    inst = instance(degree, [2, 4, 5], ["most", "one", "flow", "least"], rows_per_depth=max(40, 3 * degree))
    assert np.bincount(inst.col, minlength=inst.n).max() == degree
    same(inst)


@pytest.mark.parametrize("depth", [1, 2, 3, 4, 7, 9, 10, 11, 12, 31, 32])
@pytest.mark.parametrize("kind", ["one", "least"])
def test_tile_depths(cuda_lib, depth, kind):
    """Tiles of one depth, a full one and a remainder, of chain layers and of others."""
    same(instance(3, [depth], [kind], rows_per_depth=45))


@pytest.mark.parametrize("depths", [[1, 2, 3, 5, 8, 10], [6, 7, 13, 20, 32], [9, 10, 11]])
def test_mixed_depths_in_a_tile(cuda_lib, depths):
    same(instance(5, depths, ["one", "flow", "most", "least"], rows_per_depth=7))


@pytest.mark.parametrize("depth", [6, 7, 11, 31, 32, 33])
@pytest.mark.parametrize("kind", ["children", "three", "exactly_three"])
def test_four_node_layers(cuda_lib, depth, kind):
    """Layers of up to four nodes, alone and beside narrow rows (33 layers: the general plan)."""
    s = same(instance(3, [depth], [kind], rows_per_depth=45))
    assert s.max_width <= 4
    same(instance(6, [4, depth], [kind, "one"], rows_per_depth=20))


@pytest.mark.parametrize("depth", [33, 97, 128, 129])
def test_long_narrow_rows(cuda_lib, depth):
    """A block per tile above 32 layers; above 128 the general plan."""
    same(instance(2, [depth], ["flow", "least"], rows_per_depth=37))
    same(instance(4, [3, depth, 12], ["one", "most", "flow"], rows_per_depth=9))


@pytest.mark.parametrize("omega", [0.3, 1.0])
def test_damping(cuda_lib, omega):
    same(instance(4, [3, 6, 12], ["flow", "one"]), omega=omega)


def test_workload_shapes(cuda_lib):
    same(potts_batch(count=4, side_range=(5, 40), label_range=(2, 8), first_seed=3))
    same(sparse_matching(n_left=40, n_right=30, k=8, n_pairs=900, seed=2))


def test_zero_coefficients_and_forced_variables(cuda_lib):
    rng = np.random.default_rng(4)
    rows = []
    for _ in range(60):
        cols = np.sort(rng.choice(50, size=5, replace=False))
        vals = np.ones(5, np.int64)
        vals[rng.integers(5)] = 0
        rows.append((cols, vals, 1, SENSE_EQ))
    rows.append((np.array([50, 51]), np.array([1, 1]), 2, SENSE_EQ))  # forces both
    rows.append((np.array([3, 50]), np.array([1, 1]), 2, SENSE_LE))
    same(_from_rows("zeros", 54, rows, rng.standard_normal(54).astype(np.float32)))
