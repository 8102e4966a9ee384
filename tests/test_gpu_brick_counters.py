"""Per-brick counters: 32 bytes apart up to 4096 bricks, packed above.  The field is
a sum in whole numbers, so points in random order, which add to the counters one by
one, give the bits of the same points in grid order, which add runs; frame after
frame on one context, at the smallest grid, at the line and just above it."""

import numpy as np
import pytest

from tests import gpu_common as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("grid", [(32, 32, 32), (128, 128, 128), (128, 128, 192), (256, 128, 128)])
def test_random_order_equals_grid_order(grid, mode):
    G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    rng = np.random.default_rng(11)
    P = rng.uniform(0.02, 0.98, (7001, 3)).astype(np.float32)
    N = rng.standard_normal((7001, 3)).astype(np.float32)
    N /= np.linalg.norm(N, axis=1, keepdims=True)
    W = rng.uniform(0, 1, 7001).astype(np.float32)
    cell = np.floor(P * np.array(grid)).astype(int) // 8
    order = np.lexsort((cell[:, 0], cell[:, 1], cell[:, 2]))
    ctx = ftr.Context(grid, (0, 0, 0, 1, 1, 1), splat_mode=mode)
    fields = []
    for o in (np.arange(7001), order, np.arange(7001)):
        ctx.reset()
        ctx.splat(P[o], N[o], W[o])
        ctx.solve()
        fields.append(ctx.field_V().copy())
        assert ctx.stats()[0] == 7001
    ctx.close()
    assert np.abs(fields[0]).max() > 0
    assert np.array_equal(fields[0], fields[1]) and np.array_equal(fields[0], fields[2])
