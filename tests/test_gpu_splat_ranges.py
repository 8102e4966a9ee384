"""The splat's accumulation in each of its number ranges, against the oracle's V:
normals inside and beyond the range of the fast conversions, weights inside and
outside [0, 1], one point, one brick of several work units, and points on every
side of a brick border; weighted and simple.

Bar: every contribution is rounded to 2^-40 after a float32 product (a few
2^-24 relative), the exponentials err by a few ulps of arguments below 16
(16 * 2^-24 relative), so |V - V_oracle| <= 4e-6 max(1, |N|).
"""

import numpy as np
import pytest

from datagen import f32_box
from oracle import conventions as cv
from oracle import splat as osplat
from tests import gpu_common as G

pytestmark = pytest.mark.gpu

GRID, BOX = (32, 48, 32), (-1.0, -1.5, -1.0, 1.0, 1.5, 1.0)


def _points(kind, rng):
    n = {"one": 1, "dense": 5000, "border": 4000, "spread": 20000}[kind]
    if kind == "dense":                                  # one brick and its neighbours: several work units
        t = rng.uniform(9.0, 14.0, (n, 3))
    elif kind == "border":                               # stencils that straddle brick corners and edges
        t = 8.0 * rng.integers(1, 4, (n, 3)) + rng.uniform(-3.0, 3.0, (n, 3))
    else:
        t = rng.uniform(0.5, np.array(GRID) - 1.5, (n, 3))
    h = (np.array(BOX[3:]) - np.array(BOX[:3])) / np.array(GRID)
    return (np.array(BOX[:3]) + (t + 0.5) * h).astype(np.float32)


@pytest.mark.parametrize("mode", [cv.SPLAT_WEIGHTED, cv.SPLAT_SIMPLE])
@pytest.mark.parametrize("normal,weight", [(1.0, 1.0), (3.89, 1.0), (5.0, 1.0), (60.0, 1.0), (1.0, 3.0)])
@pytest.mark.parametrize("kind", ["one", "dense", "border", "spread"])
def test_ranges_match_the_oracle(kind, normal, weight, mode):
    G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    rng = np.random.default_rng(len(kind))
    P = _points(kind, rng)
    N = rng.standard_normal(P.shape)
    N = (normal * N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)
    W = (weight * rng.uniform(0.05, 1.0, len(P))).astype(np.float32)
    ctx = ftr.Context(GRID, BOX, splat_mode=ftr.FTR_SPLAT_WEIGHTED if mode == cv.SPLAT_WEIGHTED else ftr.FTR_SPLAT_SIMPLE)
    fields = []
    for _ in range(2):                                   # the second frame finds the accumulators cleared
        ctx.reset()
        ctx.splat(P, N, W)
        ctx.solve()
        fields.append(ctx.field_V())
    ctx.close()
    ref = osplat.splat(P, N, W, GRID, f32_box(BOX), mode=mode)
    assert np.array_equal(fields[0], fields[1])
    assert np.max(np.abs(fields[0] - ref)) <= 4e-6 * max(1.0, normal)
