"""The mesh copy into device buffers that its kernel must not store to: destinations
off the 4-byte boundary and managed memory.  They get the same bytes as a host
buffer, and nothing beside them is written."""

import ctypes

import numpy as np
import pytest

from tests import gpu_common as G

pytestmark = pytest.mark.gpu


def _mesh(ftr):
    P, N, W, _ = G.case_inputs("sphere64")
    ctx = ftr.Context((64, 64, 64), (-1.2, -1.2, -1.2, 1.2, 1.2, 1.2))
    ctx.splat(P, N, W)
    ctx.solve()
    host = ctx.mesh_numpy()
    return ctx, [host["vertices"], host["normals"], host["tris"]]


@pytest.mark.parametrize("shift", [(1, 0, 0), (0, 2, 4), (3, 3, 3)])
def test_destinations_at_any_byte(shift):
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    ctx, want = _mesh(ftr)
    buf = [torch.full((w.nbytes + s + 16,), 7, dtype=torch.uint8, device="cuda") for w, s in zip(want, shift)]
    torch.cuda.synchronize()
    ftr.ftr_mesh_copy_async(ctx.h, *[b.data_ptr() + s for b, s in zip(buf, shift)])
    torch.cuda.synchronize()
    ctx.close()
    for b, w, s in zip(buf, want, shift):
        got = b.cpu().numpy()
        assert got[s:s + w.nbytes].tobytes() == w.tobytes()
        assert np.all(got[:s] == 7) and np.all(got[s + w.nbytes:] == 7)


def test_managed_destinations():
    G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    ctx, want = _mesh(ftr)
    with open("/proc/self/maps") as f:
        cudart = ctypes.CDLL(next(line.split()[-1] for line in f if "libcudart" in line))
    cudart.cudaMallocManaged.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t, ctypes.c_uint]
    ptr = []
    for w in want:
        p = ctypes.c_void_p()
        assert cudart.cudaMallocManaged(ctypes.byref(p), w.nbytes, 1) == 0
        ptr.append(p.value)
    ftr.ftr_mesh_copy(ctx.h, *ptr)
    ctx.close()
    for p, w in zip(ptr, want):
        assert ctypes.string_at(p, w.nbytes) == w.tobytes()
        cudart.cudaFree.argtypes = [ctypes.c_void_p]
        assert cudart.cudaFree(p) == 0
