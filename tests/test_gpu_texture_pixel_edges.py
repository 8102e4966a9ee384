"""The texture stage's choice of depth pixel, floor(u + 1/2) of the float64
projection, for vertices whose projection lies on and around pixel edges and
corners, at every distance at which the kernel changes its way of deciding.  A
confidence map with a different value in every pixel shows the pixel: weights
equal to the oracle's bit for bit."""

import numpy as np
import pytest

from tests import gpu_common as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [0.0, 1e-7, 1e-6, 3e-6, 1e-5, 1e-4, 1.9e-3, 2.1e-3, 0.2, 0.45])
def test_pixel_edges(off):
    torch = G.require_gpu()
    from oracle import texture as otex
    from paper_1712_03084_gb300 import ftr
    _, _, _, views = G.case_inputs("human96")
    rng = np.random.default_rng(17)
    vs, verts = [], []
    for v in views[:3]:
        h, w = v["depth"].shape
        K, M = np.asarray(v["K"], np.float64), np.asarray(v["world_to_cam"], np.float64)
        d = dict(v)
        d["depth"] = np.full((h, w), 2.0, np.float32)
        d["conf"] = (0.25 + rng.permutation(h * w) / (2.0 * h * w)).astype(np.float32).reshape(h, w)
        vs.append(d)
        n = 400
        u = rng.integers(20, w - 20, n) + 0.5 + off * rng.choice([-1, 1], n)
        t = np.where(rng.random(n) < 0.5, rng.integers(20, h - 20, n) + 0.5 + off * rng.choice([-1, 1], n),
                     rng.uniform(20, h - 20, n))
        z = rng.uniform(0.7, 3.5, n)
        cam = np.linalg.solve(K, np.stack([u, t, np.ones(n)])) * z
        verts.append((M[:, :3].T @ (cam - M[:, 3:4])).T)
    verts = np.ascontiguousarray(np.concatenate(verts).astype(np.float32))
    n, k = len(verts), len(vs)
    dev = torch.device("cuda", 0)
    dviews = [{key: (torch.from_numpy(np.ascontiguousarray(v[key])).to(dev) if key in ("depth", "conf", "rgb")
                     else v[key]) for key in v} for v in vs]
    w = torch.zeros((n, k), device=dev)
    uv = torch.zeros((n, k, 2), device=dev)
    rgb = torch.zeros((n, 3), dtype=torch.uint8, device=dev)
    tx = torch.zeros((n,), dtype=torch.uint8, device=dev)
    ctx = ftr.Context((32, 32, 32), (0, 0, 0, 1, 1, 1))
    dv = torch.from_numpy(verts).to(dev)
    torch.cuda.synchronize()
    ftr.ftr_texture_vertices(ctx.h, dviews, 100.0, dv, w, uv, rgb, tx)
    ctx.close()
    ref = otex.texture(verts.astype(np.float64), vs, 100.0)
    assert (ref["weights"] > 0).sum() > 300
    assert np.array_equal(w.cpu().numpy(), ref["weights"].astype(np.float32))
