"""The allocation-free level at the edges of its tiling: one point, one CTA more
or less, the last size of 256 points per CTA and the next, and the largest call.

Bar: the trilinear value of one point is within a few float32 ulps of the
float64 one (its fractions are rounded once, 6e-8, and three lerps round once
each), so |L - L_oracle| <= 8 * 2^-24 max|A| for every point set; the sums run
in float64.
"""

import numpy as np
import pytest

from datagen import f32_box
from oracle import level as olevel
from tests import gpu_common as G

pytestmark = pytest.mark.gpu

GRID, BOX = (32, 48, 32), (-1.0, -1.5, -0.7, 1.3, 2.0, 1.1)
WAVE = 152 * 8 * 256                                    # points of one wave at 256 per CTA


@pytest.mark.parametrize("n", [1, 31, 255, 256, 257, 70001, WAVE, WAVE + 1, 4194304])
def test_level_sizes_match_the_oracle(n):
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    rng = np.random.default_rng(n)
    A = rng.standard_normal((GRID[2], GRID[1], GRID[0])).astype(np.float32)
    m = min(n, 70001)                                   # larger sets repeat points: the oracle sees each once
    box = np.array(f32_box(BOX))
    h = (box[3:] - box[:3]) / np.array(GRID)
    P = box[:3] + (box[3:] - box[:3]) * rng.uniform(-0.02, 1.02, (m, 3))
    near = rng.random(m) < 0.3                          # points on node planes: the decisions' edge
    P[near] = box[:3] + (np.floor((P[near] - box[:3]) / h) + 0.5) * h
    P = P.astype(np.float32)
    idx = np.arange(n) % m
    ok = olevel.osplat.accepted_mask(P, GRID, f32_box(BOX))
    val = olevel.trilinear(A, P, GRID, f32_box(BOX))
    times = np.bincount(idx, minlength=m) * ok
    want = float((val * times).sum() / times.sum()) if times.sum() else 0.0
    got = ftr.ftr_iso_level_noalloc(torch.from_numpy(A).cuda(), GRID, BOX, torch.from_numpy(P[idx]).cuda())
    assert abs(got - want) <= 8 * 2.0 ** -24 * float(np.abs(A).max())
