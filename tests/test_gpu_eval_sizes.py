"""The evaluation kernels at the edges of their tilings, against the oracle:
image sizes around the 32-row and 32-column masks, the 16 x 16 point tiles and
the SSIM tiles, dense and sparse silhouettes, overlapping and far apart.

Bars: counts, VRE and the Hausdorff distance exact (integers).  Closest-point
distances: each back-projected coordinate is rounded to float32, so a distance
moves by at most 2 sqrt(3) 2^-24 z per axis ratio r = max |X| / z of the view;
with |X| <= 2 z and z <= 4 m that is 2.8e-6 m.  WMS3IM and its terms within
1e-4 (float32 luma and window moments), as in the other appearance tests.
"""

import numpy as np
import pytest

from oracle import evaluate as oev
from tests import gpu_common as G

pytestmark = pytest.mark.gpu


def _depths(rng, w, h, kind):
    rd = np.zeros((h, w), np.float32)
    gd = np.zeros((h, w), np.float32)
    if kind == "dense":                                  # two overlapping noisy sheets
        rd[:] = 2.0 + 0.01 * rng.standard_normal((h, w))
        gd[:] = 2.0 + 0.01 * rng.standard_normal((h, w))
        rd[rng.random((h, w)) < 0.3] = 0
        gd[rng.random((h, w)) < 0.3] = 0
    elif kind == "sparse":                               # single pixels, most columns and tiles empty
        for d in (rd, gd):
            n = max(1, w * h // 400)
            d[rng.integers(0, h, n), rng.integers(0, w, n)] = rng.uniform(0.5, 4.0, n)
    else:                                                # disjoint: no pixel of one set in the other's corner
        rd[: max(1, h // 5), : max(1, w // 5)] = rng.uniform(1.0, 3.0)
        gd[h - max(1, h // 6):, w - max(1, w // 6):] = rng.uniform(1.0, 3.0)
    return rd, gd


@pytest.mark.parametrize("kind", ["dense", "sparse", "apart"])
@pytest.mark.parametrize("w,h", [(1, 1), (31, 33), (32, 32), (33, 31), (65, 64), (17, 545), (200, 15), (3, 16384)])
def test_geometry_sizes(w, h, kind):
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    rng = np.random.default_rng(w * 31 + h)
    rd, gd = _depths(rng, w, h, kind)
    f = 0.5 * max(w, h)
    K = np.array([[f, 0.01 * f, (w - 1) / 2], [0, f, (h - 1) / 2], [0, 0, 1]], np.float32)
    ctx = ftr.Context((32, 32, 32), (0, 0, 0, 1, 1, 1))
    cam = ftr.make_camera(K, np.eye(4, dtype=np.float32)[:3], w, h)
    d2 = torch.full((h, w), -1.0, device="cuda")
    torch.cuda.synchronize()
    got = ftr.ftr_eval_geometry(ctx.h, cam, torch.from_numpy(rd).cuda(), torch.from_numpy(gd).cuda(), d2)
    ctx.close()
    vre, x, o, nr, ng = oev.vre(rd, gd)
    assert (got["xor_px"], got["or_px"], got["rendered_px"], got["sensor_px"], got["vre"]) == (x, o, nr, ng, vre)
    Xg, Xr = oev.backproject(K, gd), oev.backproject(K, rd)
    assert (got["sensor_points"], got["rendered_points"]) == (len(Xg), len(Xr))
    if h < 2000:
        assert got["hausdorff_px"] == oev.hausdorff(rd, gd)
    else:                                                # the oracle's search is quadratic: a k-d tree over the pixels
        from scipy.spatial import cKDTree
        a, b = np.argwhere(rd > 0), np.argwhere(gd > 0)
        far = max((cKDTree(b).query(a)[0] ** 2).max(), (cKDTree(a).query(b)[0] ** 2).max())
        assert got["hausdorff_px"] == np.sqrt(round(far))
    d = d2.cpu().numpy()
    assert np.all(d[gd <= 0] == 0)
    step = max(1, len(Xg) // 3000)
    ref = np.sqrt(oev.closest_sq(Xg[::step], Xr))
    assert np.max(np.abs(np.sqrt(d[gd > 0])[::step] - ref)) <= 2.8e-6


@pytest.mark.parametrize("w,h", [(9, 11), (32, 16), (33, 17), (42, 26), (43, 27), (75, 53), (128, 96), (131, 77)])
def test_appearance_sizes(w, h):
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    rng = np.random.default_rng(w * 31 + h)
    v, u = np.mgrid[0:h, 0:w]
    a = (120 + 60 * np.sin(0.2 * u + 0.1 * v)[..., None] + rng.uniform(-30, 30, (h, w, 3))).astype(np.uint8)
    b = np.clip(a.astype(float) * 0.8 + rng.uniform(-20, 40, (h, w, 3)), 0, 255).astype(np.uint8)
    rd = np.where((u - w / 2) ** 2 / w ** 2 + (v - h / 2) ** 2 / h ** 2 < 0.3, 2.0, 0.0).astype(np.float32)
    ctx = ftr.Context((32, 32, 32), (0, 0, 0, 1, 1, 1))
    got = ftr.ftr_eval_appearance(ctx.h, torch.from_numpy(rd).cuda(), torch.from_numpy(a).cuda(),
                                  torch.from_numpy(b).cuda())
    none = ftr.ftr_eval_appearance(ctx.h, torch.zeros((h, w), device="cuda"), torch.from_numpy(a).cuda(),
                                   torch.from_numpy(b).cuda())
    ctx.close()
    ref, L, C, S = oev.wms3im(rd, a, b)
    assert abs(got["wms3im"] - ref) <= 1e-4
    for x, y in ((got["l"], L), (got["c"], C), (got["s"], S)):
        assert np.max(np.abs(np.array(x) - np.array(y))) <= 1e-4
    assert np.isnan(none["wms3im"])
