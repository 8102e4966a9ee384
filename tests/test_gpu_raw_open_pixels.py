"""Pixels that the raw reconstruction's float32 decisions leave open, in numbers: the
warp redoes them in float64 four at a time, a lane per triangle, in the counting pass
(a warp per 32 pixels of a row) and again in the emitting one (the tile's points, listed
densely).  Depth steps within a few ulps of the keep threshold along whole rows and
columns, in runs of two to 33 pixels, across the seams of the 32 x 16 tiles and at the
image's border, and ridges so steep that the kept unit normals nearly cancel (each
within 1.7e-4 of perpendicular to the ray, yet decided: their sum is below 1e-3).

The bars are those of the other raw tests: the point count exact, points in pixel
order within 4e-6 m, unit normals and confidences within 1e-5."""

import numpy as np
import pytest

from oracle import conventions as cv
from oracle import raw as oraw
from tests import gpu_common as G

pytestmark = pytest.mark.gpu


def _far(z0):
    """z1 > z0 whose step from z0 is the keep threshold at z1."""
    a = 3.0 * cv.TSDC_NOISE
    return (1.0 - np.sqrt(1.0 - 4.0 * a * (z0 + cv.TSDC_STEP))) / (2.0 * a)


def _ulps(z, rng):
    z = np.asarray(z, np.float32)
    return z + rng.integers(-2, 3, z.shape).astype(np.float32) * np.spacing(z)


def _depth(kind, h, w):
    rng = np.random.default_rng(h * w)
    near, far = 1.5, _far(1.5)
    d = np.zeros((h, w), np.float32)
    if kind == "rows":                                   # a step between any two rows
        d[:] = np.where(np.arange(h)[:, None] % 2 == 0, near, _ulps(np.full((h, w), far), rng))
    elif kind == "columns":                              # at both borders, at a tile's seam and inside
        side = np.zeros(w, bool)
        for c in (0, 31, 40, w - 2):
            if 0 <= c < w - 1:
                side[c + 1:] ^= True
        d[:] = np.where(side, _ulps(np.full((h, w), far), rng), near)
    elif kind == "runs":                                 # row pairs: a run in front of a run
        for k, r in enumerate(range(0, h - 1, 3)):
            m = min((2, 4, 5, 6, 9, 32, 33)[k % 7], w)
            u = min((0, 31, 27, w - m, 28, 32, 60)[(k + k // 7) % 7], w - m)
            d[r, u:u + m] = near
            d[r + 1, u:u + m] = _ulps(np.full(m, far), rng)
    else:                                                # ridges and valleys along the columns, rows alike
        d[:] = near + 0.03 * np.abs((np.arange(w) + 4) % 8 - 4)
    return d


def _open_pixels(d):
    """Per pixel, whether the depth-step test of one of its six triangles is open in float32."""
    f = np.float32
    quad = [d[:-1, :-1], d[:-1, 1:], d[1:, :-1], d[1:, 1:]]
    out = np.zeros(d.shape, bool)
    for tri in ((0, 1, 2), (1, 3, 2)):
        z = np.stack([quad[i] for i in tri])
        thr = (f(cv.TSDC_STEP) + f(3.0) * f(cv.TSDC_NOISE) * z.max(0) * z.max(0)).astype(f)
        und = (z > 0).all(0) & (np.abs((z.max(0) - z.min(0)) - thr) <= f(1e-5) * thr)
        for i in tri:
            out[i // 2:i // 2 + und.shape[0], i % 2:i % 2 + und.shape[1]] |= und
    return out


@pytest.mark.parametrize("shape", [(2, 33), (17, 64), (47, 97)])
@pytest.mark.parametrize("kind", ["rows", "columns", "runs", "ridges"])
def test_open_pixels_equal_the_oracle(kind, shape):
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    h, w = shape
    d = _depth(kind, h, w)
    f = 400000.0 if kind == "ridges" else 400.0
    K = np.array([[f, 0.0, w / 2], [0.0, f, h / 2], [0.0, 0.0, 1.0]])
    M = np.eye(4)[:3]
    if kind != "ridges":
        pad = np.zeros((h, -w % 32), bool)
        per_warp = np.concatenate([_open_pixels(d), pad], 1).reshape(h, -1, 32).sum(2)
        assert per_warp.max() >= {"rows": 32, "columns": 2, "runs": min(w, 32) if h > 17 else 2}[kind]
        if kind == "runs" and h > 17:
            assert {1, 2, 4, 5, 32} <= set(np.unique(per_warp))
    else:
        total = np.zeros((h, w, 3))
        for corners, _, n in oraw.triangle_normals(oraw.camera_points(d, K), d):
            for a, b in corners:
                total[a:a + h - 1, b:b + w - 1] += n
        cancel = (total ** 2).sum(-1)
        assert ((cancel > 1e-7) & (cancel < 9e-7)).sum() >= h - 2 and not ((cancel >= 9e-7) & (cancel < 0.1)).any()
    P, N, W, conf_ref = oraw.raw_points(d, K, M)
    conf = torch.full((h, w), -1.0, device="cuda")
    ctx = ftr.Context((64, 64, 64), np.array([-4, -4, -4, 4, 4, 4], np.float32))
    ctx.reset()
    ftr.ftr_splat_depth(ctx.h, [{"depth": torch.from_numpy(d).cuda(), "K": K, "world_to_cam": M}], conf_out=[conf])
    n = ctx.stats()[0]
    buf = np.zeros(7 * d.size, np.float32)
    ftr.ftr_debug_buffer(ctx.h, 2, buf)
    ctx.close()
    px = d.size
    assert n == len(P)
    assert np.abs(buf[:3 * n].reshape(-1, 3) - P).max(initial=0) <= 4e-6
    assert np.abs(buf[3 * px:3 * px + 3 * n].reshape(-1, 3) - N).max(initial=0) <= 1e-5
    assert np.abs(buf[6 * px:6 * px + n] - W).max(initial=0) <= 1e-5
    assert np.abs(conf.cpu().numpy() - conf_ref).max() <= 1e-5
