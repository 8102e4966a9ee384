"""Rows of V without a touched brick are skipped by the x and y passes: the same
V given densely (every row transformed) must yield the same indicator, bit for
bit, for sparse point sets (two far clusters with a gap along y, one brick, a
cluster at the grid's edge, no point) in every tile plan and precision, also
right after a frame that filled other rows.
"""

import numpy as np
import pytest

from tests import gpu_common as G

pytestmark = pytest.mark.gpu


def _points(kind, grid, rng):
    centres = {"gap": [(0.3, 0.15, 0.3), (0.6, 0.85, 0.7)], "one": [(0.5, 0.52, 0.5)],
               "edge": [(0.5, 0.97, 0.03)], "none": []}[kind]
    n = np.array(grid)
    pts = [np.array(c) * n + rng.uniform(-2.5, 2.5, (300, 3)) for c in centres] or [np.zeros((0, 3))]
    P = (np.concatenate(pts) + 0.5) / n                # unit box, one node per 1 / n
    N = rng.standard_normal(P.shape)
    return P.astype(np.float32), N.astype(np.float32), rng.uniform(0, 1, len(P)).astype(np.float32)


@pytest.mark.parametrize("kind", ["gap", "one", "edge", "none"])
@pytest.mark.parametrize("grid,prec,plans", [
    ((64, 64, 64), 0, [(8, 8, 8), (16, 16, 16), (32, 32, 32), (-16, -16, 16)]),
    ((48, 96, 48), 0, [(16, 16, 16), (-16, -16, 8)]),
    ((32, 384, 32), 0, [(8, 16, 16), (16, 16, 16)]),
    ((64, 128, 256), 0, [(16, 16, 16), (-16, 16, 16)]),
    ((64, 128, 64), 1, [None]), ((128, 64, 64), 2, [None]), ((64, 384, 64), 1, [None]),
])
def test_sparse_rows_equal_dense_rows(grid, prec, plans, kind):
    G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    rng = np.random.default_rng(7)
    P, N, W = _points(kind, grid, rng)
    Q = rng.uniform(0.1, 0.9, (3000, 3)).astype(np.float32)     # an earlier frame that touches most rows
    ctx = ftr.Context(grid, (0, 0, 0, 1, 1, 1), precision=prec)
    for plan in plans:
        if plan:
            ctx.set_plan(plan)
        ctx.reset()
        ctx.splat(Q, Q, None)
        ctx.solve()
        ctx.reset()
        ctx.splat(P, N, W)
        ctx.solve()
        A, V = ctx.field_A(), ctx.field_V()
        ctx.reset()
        ctx.set_field_V(V)
        ctx.solve()
        assert np.array_equal(A, ctx.field_A())
        assert kind == "none" or np.abs(A).max() > 0
    ctx.close()
