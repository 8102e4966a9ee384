"""Split-precision solves are the same bits every time: line maxima, operand
buffers and tables shared by a thread block are ordered by its barriers, whichever
warp comes first.  Every axis length of each pass, ten solves, no tolerance."""

import numpy as np
import pytest

from tests import gpu_common as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("grid", [(64, 128, 256), (384, 64, 128), (128, 384, 64), (256, 64, 384)])
def test_repeated_solves_are_equal(grid, prec):
    G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    rng = np.random.default_rng(5)
    d = rng.standard_normal((4000, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    P = (0.5 + 0.3 * d).astype(np.float32)
    ctx = ftr.Context(grid, (0, 0, 0, 1, 1, 1), precision=prec)
    first = None
    for _ in range(10):
        ctx.reset()
        ctx.splat(P, d.astype(np.float32), np.ones(len(P), np.float32))
        ctx.solve()
        A = ctx.field_A()
        if first is None:
            first = A.copy()
            assert np.isfinite(first).all() and first.max() > first.min()
        assert np.array_equal(A, first)
    ctx.close()
