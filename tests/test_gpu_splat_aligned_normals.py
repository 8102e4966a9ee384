"""Normals longer than one, all the same way and close to one grid node: the sums
of one work unit grow to its 1024 pairs times the component, beyond the 32-bit
halves that unit normals fit in, where isotropic directions would cancel.
Weighted and simple, against the oracle's V.

Bar: that of the other range tests -- every contribution is rounded to 2^-40
after a float32 product (a few 2^-24 relative), the exponentials err by a few
ulps -- so |V - V_oracle| <= 4e-6 max(1, |N|)."""

import numpy as np
import pytest

from datagen import f32_box
from oracle import conventions as cv
from oracle import splat as osplat
from tests import gpu_common as G

pytestmark = pytest.mark.gpu

GRID, BOX = (32, 48, 32), (-1.0, -1.5, -1.0, 1.0, 1.5, 1.0)


@pytest.mark.parametrize("mode", [cv.SPLAT_WEIGHTED, cv.SPLAT_SIMPLE])
@pytest.mark.parametrize("nz", [1.0, 1.98, 2.0, -2.5, 3.8, 60.0, -60.0])
@pytest.mark.parametrize("n", [40, 1024, 5000])
def test_sums_of_aligned_normals(n, nz, mode):
    G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    rng = np.random.default_rng(n)
    t = np.array([12.0, 19.0, 11.0]) + rng.uniform(-0.15, 0.15, (n, 3))      # node units, inside one brick
    P = (np.array(BOX[:3]) + (t + 0.5) * (np.array(BOX[3:]) - np.array(BOX[:3])) / np.array(GRID)).astype(np.float32)
    N = np.tile(np.array([0.0, 0.25 * nz, nz], np.float32), (n, 1))
    W = np.ones(n, np.float32)
    ctx = ftr.Context(GRID, BOX, splat_mode=ftr.FTR_SPLAT_WEIGHTED if mode == cv.SPLAT_WEIGHTED else ftr.FTR_SPLAT_SIMPLE)
    ctx.splat(P, N, W)
    ctx.solve()
    V = ctx.field_V()
    ctx.close()
    ref = osplat.splat(P, N, W, GRID, f32_box(BOX), mode=mode)
    assert np.max(np.abs(ref)) > 0.5 * abs(nz)
    assert np.max(np.abs(V - ref)) <= 4e-6 * max(1.0, abs(nz))
