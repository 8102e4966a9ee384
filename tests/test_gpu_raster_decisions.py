"""The rasteriser's float32 shortcuts against the float64 oracle, bit for bit, on
triangles chosen to land on its decisions: vertices exactly on pixel centres
(edges through centres), slivers, edge-on and zero-area triangles, vertices
nearer than the near plane or behind the camera, projections far outside the
image and too large for float32, many triangles over the same pixels (more
fragments than a CTA queues) and large triangles; with and without skew.
Depths are decided in one fixed float64 order on both sides: equality.
"""

import numpy as np
import pytest

from oracle import render as orender
from tests import gpu_common as G

pytestmark = pytest.mark.gpu

W, H = 61, 47


def _mesh(kind, rng, K):
    n = 256

    def back(u, v, z):                                  # world = camera coordinates
        y = (v - K[1, 2]) / K[1, 1]
        x = (u - K[0, 2] - K[0, 1] * y) / K[0, 0]
        return np.stack([x * z, y * z, z], -1)
    u, v = rng.uniform(-8, W + 8, (n, 3)), rng.uniform(-8, H + 8, (n, 3))
    z = rng.uniform(0.5, 4.0, (n, 3))
    if kind == "centres":                               # integer pixel positions, equal depths: ties by index
        u, v, z = np.round(u), np.round(v), np.repeat(np.round(z[:, :1]), 3, 1)
    elif kind == "small":                               # around one pixel
        u, v = u[:, :1] + rng.uniform(-0.8, 0.8, (n, 3)), v[:, :1] + rng.uniform(-0.8, 0.8, (n, 3))
    elif kind == "slivers":
        t = rng.uniform(0, 1, (n, 1))
        u[:, 2:], v[:, 2:] = u[:, :1] * t + u[:, 1:2] * (1 - t), v[:, :1] * t + v[:, 1:2] * (1 - t)
        u[:, 2] += rng.choice([0.0, 1e-7, 1e-4, 0.05], n)
    elif kind == "edge_on":                             # the plane passes (almost) through the camera centre
        z = rng.uniform(0.5, 30.0, (n, 3))
        u, v = u[:, :1] + rng.uniform(-0.05, 0.05, (n, 3)), v[:, :1] + rng.uniform(-6, 6, (n, 3))
    elif kind == "near":
        z = rng.choice([-1.0, 0.0, 0.00999, 0.01, 0.011, 1.0, 2.0], (n, 3))
    elif kind == "wild":
        far = rng.random((n, 3)) < 0.3
        u, v = np.where(far, u * 10.0 ** rng.integers(3, 9, (n, 3)), u), np.where(far, v * 1e5, v)
    elif kind == "piled":                               # every triangle covers the same 25 x 25 pixels
        u = np.tile([[10.0, 60.0, 10.0]], (n, 1)) + rng.uniform(0, 1, (n, 3))
        v = np.tile([[5.0, 5.0, 45.0]], (n, 1)) + rng.uniform(0, 1, (n, 3))
    P = back(u, v, z)
    return P.reshape(-1, 3).astype(np.float32), np.arange(3 * n, dtype=np.int32).reshape(n, 3)


@pytest.mark.parametrize("skew", [0.0, 0.7])
@pytest.mark.parametrize("kind", ["any", "centres", "small", "slivers", "edge_on", "near", "wild", "piled"])
def test_depth_is_bit_exact(kind, skew):
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    rng = np.random.default_rng(len(kind))
    K = np.array([[64.0, skew, 30.0], [0, 64.0, 23.0], [0, 0, 1]], np.float32)
    RT = np.eye(4, dtype=np.float32)[:3]
    verts, tris = _mesh(kind, rng, K.astype(np.float64))
    tris = np.concatenate([tris, tris[::-1][:, [0, 2, 1]], [[0, 1, len(verts)], [0, -1, 2]]]).astype(np.int32)
    ctx = ftr.Context((32, 32, 32), (0, 0, 0, 1, 1, 1))
    depth = torch.full((H, W), -1.0, device="cuda")
    torch.cuda.synchronize()
    ftr.ftr_render(ctx.h, torch.from_numpy(verts).cuda(), torch.from_numpy(tris).cuda(), ftr.make_camera(K, RT, W, H),
                   depth)
    ctx.close()
    with np.errstate(all="ignore"):
        ref, win = orender.rasterise(verts, tris[:-2], K, RT, W, H)
    assert np.array_equal(depth.cpu().numpy(), ref)
    assert (win >= 0).any() or kind == "edge_on"
