"""n_vertices as no more than a bound on the indices: the vertices past the array's end
are neither read nor given scratch (the vertices lie at the end of an allocation of
their own), and the depth is that of the exact count, bit for bit.  Which way a call
took shows in its launches: clear aside, projection, two raster passes and resolve,
or the last three."""

import ctypes

import numpy as np
import pytest

from tests import gpu_common as G

pytestmark = pytest.mark.gpu

W, H = 80, 60


@pytest.mark.parametrize("scale", [1.0, 0.02])           # large triangles; small ones
def test_vertices_past_the_array_are_not_touched(scale):
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    rng = np.random.default_rng(5)
    nt, nv = 700, 500
    verts = rng.uniform(-1, 1, (nv, 3)).astype(np.float32) + np.array([0, 0, 3], np.float32)
    tris = rng.integers(0, nv, (nt, 3)).astype(np.int32)
    verts[tris[:, 1]] = verts[tris[:, 0]] + scale * rng.uniform(-1, 1, (nt, 3)).astype(np.float32)
    K = np.array([[60.0, 0, 40], [0, 60.0, 30], [0, 0, 1]], np.float32)
    cam = ftr.make_camera(K, np.eye(4, dtype=np.float32)[:3], W, H)
    dev_tris = torch.from_numpy(tris).cuda()
    depth = torch.zeros((H, W), device="cuda")
    torch.cuda.synchronize()
    with open("/proc/self/maps") as f:
        cudart = ctypes.CDLL(next(line.split()[-1] for line in f if "libcudart" in line))
    cudart.cudaMalloc.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t]
    cudart.cudaMemcpy.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]
    cudart.cudaFree.argtypes = [ctypes.c_void_p]
    own = ctypes.c_void_p()
    assert cudart.cudaMalloc(ctypes.byref(own), verts.nbytes) == 0
    assert cudart.cudaMemcpy(own, verts.ctypes.data, verts.nbytes, 1) == 0
    ctx = ftr.Context((32, 32, 32), (0, 0, 0, 1, 1, 1))

    def render(n):
        depth.fill_(-1.0)
        torch.cuda.synchronize()
        before = ctx.launch_count()
        ftr.ftr_render(ctx.h, own.value, dev_tris, cam, depth, n_vertices=n)
        ftr.ftr_stats(ctx.h)                             # waits for the context's stream
        torch.cuda.synchronize()
        return depth.cpu().numpy(), ctx.launch_count() - before

    want, launches = render(nv)
    assert launches == 4 and (want > 0).any()
    # inside the triangles' bound but past the allocation; past the bound; beyond any memory
    for n in (3 * nt, 3 * nt + 1, 10 ** 7, 2 ** 40):
        got, launches = render(n)
        assert launches == 3 and np.array_equal(got, want)
    ctx.close()
    assert cudart.cudaFree(own) == 0
