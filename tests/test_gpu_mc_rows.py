"""Marching cubes with row classes (rows wholly outside or inside are taken from
their class): fields whose surface lies on, beside and between such rows, on
every word count per row and tile size, against the oracle's mesh: equal vertex
and triangle counts, equal triangles, vertices within a few float32 ulps of the
box; and the inside mask against A >= L.
"""

import numpy as np
import pytest

from datagen import f32_box
from oracle import mc as omc
from tests import gpu_common as G

pytestmark = pytest.mark.gpu

BOX = (-1.0, -0.5, -2.0, 1.0, 1.5, 2.0)


def _field(kind, grid, rng):
    nx, ny, nz = grid
    z, y, x = np.meshgrid(*(np.arange(n) for n in (nz, ny, nx)), indexing="ij")
    if kind == "slab":                                   # whole planes inside, none mixed
        A = np.where((z > nz // 3) & (z < nz // 2), 1.0, 0.0)
    elif kind == "rows":                                 # single rows inside, first and last among them
        A = np.where(((y + 3 * z) % 17 == 0) | ((y == ny - 1) & (z == nz - 1)), 1.0, -1.0)
    elif kind == "column":                               # one node column at the x border
        A = np.where((x == nx - 1) & (y == 5) & (z > 2), 2.0, -1.0)
    elif kind == "nodes":                                # a few single nodes
        A = np.full((nz, ny, nx), -1.0)
        A.reshape(-1)[rng.integers(0, A.size, 9)] = 1.0
    elif kind == "inside":
        A = np.ones((nz, ny, nx))
    else:                                                # every row mixed
        A = np.sin(0.9 * x + 0.3) * np.cos(0.5 * y) + 0.3 * np.sin(0.7 * z) + 0.01 * rng.standard_normal((nz, ny, nx))
    return np.ascontiguousarray(A.astype(np.float32))


@pytest.mark.parametrize("tile", [128, 256, 512])
@pytest.mark.parametrize("grid", [(32, 32, 32), (48, 32, 64), (96, 48, 32), (384, 32, 32), (512, 32, 32)])
@pytest.mark.parametrize("kind", ["slab", "rows", "column", "nodes", "inside", "waves"])
def test_row_classes_keep_the_mesh(kind, grid, tile):
    G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    A = _field(kind, grid, np.random.default_rng(3))
    L = 0.25
    ctx = ftr.Context(grid, BOX)
    ctx.set_mc_plan((tile, 4))
    ctx.set_indicator(np.full_like(A, -5.0), 0.0)        # leaves no surface: state of a frame before
    ctx.mesh_numpy()
    ctx.set_indicator(A, L)
    got = ctx.mesh_numpy()
    mask = ctx.inside_mask()
    ctx.close()
    ref = omc.marching_cubes(A.astype(np.float64), L, grid, f32_box(BOX))
    assert np.array_equal(mask, A >= L)
    assert np.array_equal(got["tris"], ref["tris"])
    assert got["vertices"].shape == ref["vertices"].shape
    if len(ref["vertices"]):
        assert np.max(np.abs(got["vertices"] - ref["vertices"])) <= 8 * 2.0 ** -24 * 2.0
