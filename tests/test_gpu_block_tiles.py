"""Block tiles with one barrier a layer (min-sum solvers, layers of at most 512 nodes) at the edges of their
forms -- one, two and four nodes per thread, the widest layer they take and one wider, single layers,
merged nodes with many predecessors -- against the persistent schedule, whose block tiles are the
general form: the same multipliers and pending sums bit for bit, bounds up to the order of their FP64
sums; min-marginals against the oracle (1e-5, the parity tests' bound for FP32 path sums)."""
from __future__ import annotations

import numpy as np
import pytest

from instances import SENSE_EQ, SENSE_LE
from instances.generators import _from_rows
from oracle import Oracle

pytestmark = pytest.mark.gpu


def cardinality(width, seed=0):
    """One at-most-half row whose widest layer has `width` nodes, and narrow rows beside it."""
    rng = np.random.default_rng([seed, width])
    n = 2 * (width - 1)
    rows = [(np.arange(n), np.ones(n), width - 1, SENSE_LE)]
    for k in (2, 3, 5, 17, 33):
        rows.append((np.sort(rng.choice(n, size=min(k, n), replace=False)), np.ones(min(k, n)), min(k, n) // 2 + 1, SENSE_LE))
    return _from_rows(f"cardinality_{width}", n, rows, rng.standard_normal(n).astype(np.float32))


def weighted(n, top, sense, seed=0):
    """Rows with coefficients up to `top`: nodes merge, some with many predecessors."""
    rng = np.random.default_rng([seed, n, top])
    rows = []
    for _ in range(6):
        k = int(rng.integers(n // 2, n + 1))
        cols = np.sort(rng.choice(n, size=k, replace=False))
        vals = rng.integers(1, top + 1, size=k) * np.where(rng.random(k) < 0.2, -1, 1)
        rows.append((cols, vals, int(vals[rng.random(k) < 0.5].sum()), sense))
    return _from_rows(f"weighted_{n}_{top}", n, rows, rng.standard_normal(n).astype(np.float32))


def check(inst, iters=11, **kw):
    import torch

    from paper_2009_00481_gb300 import Solver
    out = []
    for schedule in (1, 0):
        s = Solver(inst, schedule=schedule, **kw)
        t = torch.zeros(iters, dtype=torch.float64, device="cuda")
        s.iterate_device(iters, trace=t)
        torch.cuda.synchronize()
        out.append((s, t.cpu().numpy(), s.get_state()))
    (a, ta, (la, pa)), (_, tb, (lb, pb)) = out
    assert np.all(np.abs(ta - tb) <= 1e-12 * np.maximum(1.0, np.abs(tb)))
    np.testing.assert_array_equal(la, lb)
    np.testing.assert_array_equal(pa, pb)
    _, _, m0, m1 = a.iterate(0, mm=True)
    o = Oracle(inst)
    o.set_state(la.astype(np.float64), pa.astype(np.float64))
    for got, want in zip((m0, m1), o.min_marginals(fold=True)):
        fin = np.isfinite(want)
        np.testing.assert_array_equal(np.isfinite(got), fin)
        assert np.all(np.abs(got[fin] - want[fin]) <= 1e-5 * np.maximum(1.0, np.abs(want[fin])))
    return a


@pytest.mark.parametrize("width", [33, 64, 127, 128, 129, 255, 256, 257, 511, 512, 513])
def test_widths(cuda_lib, width):
    s = check(cardinality(width))
    assert s.max_width == width and s.block_tiles >= 1


@pytest.mark.parametrize("sense", [SENSE_LE, SENSE_EQ])
@pytest.mark.parametrize("n,top", [(40, 5), (24, 40), (90, 3)])
def test_weighted_rows(cuda_lib, n, top, sense):
    check(weighted(n, top, sense))


@pytest.mark.parametrize("depth", [1, 2, 3, 7, 8, 9, 40])
def test_pieces(cuda_lib, depth):
    """Sub-BDDs: several roots, copy arcs in the last layer, pieces of a single layer; their bounds
    against the oracle's (1e-4, the split parity tests' bound)."""
    import torch

    from paper_2009_00481_gb300 import Solver
    inst = cardinality(70, seed=3)
    s = Solver(inst, split_depth=depth)
    t = torch.zeros(20, dtype=torch.float64, device="cuda")
    s.iterate_device(20, trace=t)
    o = Oracle(inst)
    o.split_depth(depth)
    want = o.run_parallel(20, omega=0.5)
    assert np.all(np.abs(t.cpu().numpy() - want) <= 1e-4 * np.maximum(1.0, np.abs(want)))
