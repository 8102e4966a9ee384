"""A solve that stopped half way leaves nothing behind for the next one.

Every launch reports the calling thread's last CUDA error, also one that the
application left there (here: an allocation that cannot succeed).  A solve that
meets one has enqueued its binning but not its accumulation; the next solve,
with or without a reset between, and the next queued frame give what a fresh
context gives, bit for bit (the grids have more bricks with points than not,
where stale unit counts reach farthest)."""

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


@pytest.mark.parametrize("how", ["reset", "again", "frame"])
@pytest.mark.parametrize("n", [64, 32])
def test_solve_after_a_failed_solve(n, how):
    G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    first, second = _points(30000, 1), _points(20000, 2)
    want = second if how == "reset" else first
    fresh = ftr.Context((n, n, n), BOX)
    fresh.splat(*want)
    level = fresh.solve()
    V, A = fresh.field_V(), fresh.field_A()
    fresh.close()

    ctx = ftr.Context((n, n, n), BOX)
    ctx.splat(*first)
    _leave_error()
    with pytest.raises(ftr.FtrError):
        ctx.solve()
    if how == "reset":
        ctx.reset()
        ctx.splat(*second)
    if how == "frame":
        ftr.ftr_frame_launch(ctx.h, [], 0.0, 0)
        ftr.ftr_frame_finish(ctx.h)
    else:
        assert ctx.solve() == level
    assert np.array_equal(ctx.field_V(), V) and np.array_equal(ctx.field_A(), A)
    for _ in range(2):                                   # and the frames after it
        ctx.reset()
        ctx.splat(*want)
        assert ctx.solve() == level
    assert np.array_equal(ctx.field_V(), V)
    ctx.close()
