"""A splat call that fails has counted nothing: called again, without a reset, the
frame is a fresh context's, bit for bit.  (The error is one that the application
left on the calling thread, an allocation that cannot succeed, which every call
that launches reports.)"""

import ctypes

import numpy as np
import pytest

from tests import gpu_common as G

pytestmark = pytest.mark.gpu

BOX = (-1.2, -1.2, -1.2, 1.2, 1.2, 1.2)


def _leave_error():
    """An allocation of 2^60 bytes on the runtime that the library uses: refused,
    and kept as the thread's last error."""
    with open("/proc/self/maps") as f:
        path = next(line.split()[-1] for line in f if "libcudart" in line)
    p = ctypes.c_void_p()
    cudart = ctypes.CDLL(path)
    cudart.cudaMalloc.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t]
    assert cudart.cudaMalloc(ctypes.byref(p), 1 << 60) != 0


def _points(n, seed):
    rng = np.random.default_rng(seed)
    P = rng.uniform(-1.1, 1.1, (n, 3)).astype(np.float32)
    N = rng.standard_normal((n, 3))
    N = (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)
    return P, N, rng.uniform(0.1, 1.0, n).astype(np.float32)


@pytest.mark.parametrize("how", ["points", "sets", "host"])
def test_splat_again_after_a_failed_one(how):
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    pts = _points(30000, 3)
    arrays = pts if how == "host" else [torch.from_numpy(a).cuda() for a in pts]
    torch.cuda.synchronize()

    def splat(ctx):
        if how == "sets":
            ftr.ftr_splat_sets(ctx.h, [tuple(a[:9999] for a in arrays), tuple(a[9999:] for a in arrays)])
        else:
            ctx.splat(*arrays)

    fresh = ftr.Context((64, 64, 64), BOX)
    splat(fresh)
    level, V = fresh.solve(), fresh.field_V()
    fresh.close()
    ctx = ftr.Context((64, 64, 64), BOX)
    _leave_error()
    with pytest.raises(ftr.FtrError):
        splat(ctx)
    splat(ctx)
    assert ctx.stats() == (len(pts[0]), 0)
    assert ctx.solve() == level and np.array_equal(ctx.field_V(), V)
    ctx.close()
