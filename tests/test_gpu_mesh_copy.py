"""The one-launch mesh copy into device buffers: destinations at every 4-byte
alignment, any of the three left out, nothing written past the mesh; equal to
the copies into host memory.  After ftr_reset the counters of the frame before
are gone (points, dropped points, wide weights)."""

import numpy as np
import pytest

from tests import gpu_common as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("skip", [(), (0,), (1, 2), (0, 1, 2)])
@pytest.mark.parametrize("shift", [0, 1, 3])
def test_device_copies_equal_host_copies(shift, skip):
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    P, N, W, _ = G.case_inputs("sphere64")
    ctx = ftr.Context((64, 64, 64), (-1.2, -1.2, -1.2, 1.2, 1.2, 1.2))
    ctx.splat(P, N, W)
    ctx.solve()
    host = ctx.mesh_numpy()
    want = [host["vertices"], host["normals"], host["tris"]]
    flat = [torch.full((w.size + shift + 8,), 7, dtype=torch.int32 if w.dtype == np.int32 else torch.float32,
                       device="cuda") for w in want]
    dst = [None if i in skip else f[shift:shift + w.size].reshape(-1, 3) for i, (f, w) in enumerate(zip(flat, want))]
    torch.cuda.synchronize()
    ftr.ftr_mesh_copy_async(ctx.h, *dst)
    torch.cuda.synchronize()
    for i, (f, w) in enumerate(zip(flat, want)):
        got = f.cpu().numpy()
        body = got[shift:shift + w.size].reshape(w.shape)
        assert np.all(body == 7) if i in skip else np.array_equal(body, w)
        assert np.all(got[:shift] == 7) and np.all(got[shift + w.size:] == 7)
    ctx.close()


def test_reset_clears_the_frames_counters():
    G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    P, N, W, _ = G.case_inputs("sphere64")
    ctx = ftr.Context((64, 64, 64), (-1.2, -1.2, -1.2, 1.2, 1.2, 1.2))
    ctx.splat(P, N, W)
    level = ctx.solve()
    A = ctx.field_A()
    ctx.reset()
    ctx.splat(P * 3.0, N, 5.0 * W)                       # most points outside, weights beyond [0, 1]
    ctx.solve()
    assert ctx.stats()[1] > len(P) // 2
    ctx.reset()
    assert ctx.stats() == (0, 0)
    ctx.splat(P, N, W)
    assert ctx.solve() == level and np.array_equal(ctx.field_A(), A)
    assert ctx.stats() == (len(P), 0)
    ctx.close()
