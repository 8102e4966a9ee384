"""The texture stage at the edges of its tiling: every camera count 1..8 and
vertex counts around a CTA's share (256 / G vertices), against the oracle.

Bars as in the other texture tests: weights bit-equal, UVs within 1e-3 px,
flags equal, colours within 1 LSB.  Outputs one entry longer than the vertices
stay untouched past them, and may be missing.
"""

import numpy as np
import pytest

from tests import gpu_common as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,n", [(1, 255), (1, 257), (2, 128), (3, 65), (4, 63), (4, 1), (5, 33), (6, 32), (7, 31),
                                 (8, 97)])
def test_camera_counts_and_vertex_tails(k, n):
    torch = G.require_gpu()
    from oracle import texture as otex
    from paper_1712_03084_gb300 import ftr
    _, _, _, views = G.case_inputs("human96")
    views = [views[i % len(views)] for i in range(k)]
    P = G.case_inputs("human96")[0]
    verts = np.ascontiguousarray(P[np.random.default_rng(k).permutation(len(P))[:n]])
    dev = torch.device("cuda", 0)
    dviews = [{key: (torch.from_numpy(np.ascontiguousarray(v[key])).to(dev) if key in ("depth", "conf", "rgb")
                     else v[key]) for key in v} for v in views]
    w = torch.full((n + 1, k), 7.0, device=dev)
    uv = torch.full((n + 1, k, 2), 7.0, device=dev)
    rgb = torch.full((n + 1, 3), 7, dtype=torch.uint8, device=dev)
    tx = torch.full((n + 1,), 7, dtype=torch.uint8, device=dev)
    tol = float(np.float32(0.03))
    ctx = ftr.Context((32, 32, 32), (0, 0, 0, 1, 1, 1))
    dv = torch.from_numpy(verts).to(dev)
    torch.cuda.synchronize()
    ftr.ftr_texture_vertices(ctx.h, dviews, tol, dv, w, uv, rgb, tx)
    ftr.ftr_texture_vertices(ctx.h, dviews, tol, dv, None, None, None, tx)
    ctx.close()
    ref = otex.texture(verts.astype(np.float64), views, tol)
    got = [t.cpu().numpy() for t in (w, uv, rgb, tx)]
    assert all(np.all(g[n] == 7) for g in got)
    vis = ref["weights"] > 0
    assert vis.any()
    assert np.array_equal(got[0][:n], ref["weights"].astype(np.float32))
    assert np.max(np.abs(got[1][:n][vis] - ref["uv"][vis])) <= 1e-3
    assert np.all(got[1][:n][~vis] == -1)
    assert np.max(np.abs(got[2][:n].astype(int) - ref["rgb"].astype(int))) <= 1
    assert np.array_equal(got[3][:n], ref["textured"])
