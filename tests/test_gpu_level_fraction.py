"""The fraction of a point between its nodes, as the allocation-free level takes
it: rounded once.  An indicator that alternates 0, 1 along x makes the level of
a single point behind an even node exactly that fraction (the lerps along y and
z are between equal values).

Bar: the rounding of the fraction itself, 2^-24 of it, or 2^-25 where it is one
less a small remainder, plus 1e-10 for the float pair that the position is formed
in (its error is below 1e-11 for coordinates under 512)."""

import numpy as np
import pytest

from datagen import f32_box
from tests import gpu_common as G

pytestmark = pytest.mark.gpu


def _coordinates(nx, lo, hi, n, rng):
    """Float32 x behind even nodes: anywhere, just before the next node, just
    behind the node (where the float product can still lie before it)."""
    h = (hi - lo) / nx
    node = 2.0 * rng.integers(1, nx // 2 - 2, n)
    near = 10.0 ** rng.uniform(-5.9, -4.2, n)
    frac = np.choose(rng.integers(0, 3, n), [rng.random(n), 1.0 - near, near])
    x = (lo + (node + frac + 0.5) * h).astype(np.float32)
    t = (x.astype(np.float64) - lo) / h - 0.5
    keep = np.floor(t) % 2 == 0
    return x[keep], (t - np.floor(t))[keep]


@pytest.mark.parametrize("nx", [64, 256, 512])
def test_fraction_is_rounded_once(nx):
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    grid, box = (nx, 32, 32), (-1.37, -1.0, -1.0, 2.11, 1.0, 1.0)
    b = f32_box(box)
    x, want = _coordinates(nx, b[0], b[3], 3000, np.random.default_rng(nx))
    P = np.zeros((len(x), 3), np.float32)
    P[:, 0] = x
    P = torch.from_numpy(P).cuda()
    A = torch.from_numpy(np.broadcast_to(np.arange(nx, dtype=np.float32) % 2, (32, 32, nx)).copy()).cuda()
    got = np.array([ftr.ftr_iso_level_noalloc(A, grid, box, P[i:i + 1]) for i in range(len(x))])
    bar = np.where(want > 0.99, 2.0 ** -25, 2.0 ** -24 * want) + 1e-10
    assert np.max(np.abs(got - want) - bar) <= 0.0
