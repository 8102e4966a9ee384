"""Raw reconstruction at the edges of its tiles and windows: widths around the
256 pixels of a tile and the 32 of a mask word, points at the image's border,
rows without a foreground pixel, the smallest and largest W2 windows."""

import numpy as np
import pytest

from oracle import raw as oraw
from tests import gpu_common as G

pytestmark = pytest.mark.gpu


def _depth(h, w, seed):
    """A tilted, gently curved surface (depth steps of ~1 mm a pixel, far from
    the 30 mm keep threshold) over a random silhouette of runs, with empty rows
    and isolated pixels."""
    rng = np.random.default_rng(seed)
    v, u = np.mgrid[0:h, 0:w].astype(np.float64)
    d = 1.5 + 0.0004 * u + 0.0007 * v + 0.002 * np.sin(0.21 * u) * np.cos(0.17 * v)
    keep = np.repeat(rng.random((h, (w + 6) // 7)) < 0.6, 7, axis=1)[:, :w]
    keep |= rng.random((h, w)) < 0.02
    keep[h // 3: h // 3 + 3] = False
    return np.where(keep, d, 0.0).astype(np.float32)


@pytest.mark.parametrize("radius", [0, 10, 16])
@pytest.mark.parametrize("shape", [(2, 2), (5, 31), (9, 33), (40, 255), (3, 256), (21, 257), (17, 520)])
def test_points_and_confidence_equal_the_oracle(shape, radius):
    """The point count is exact, points in pixel order within 4e-6 m, unit
    normals within 1e-5, confidences within 1e-5 (float32 kernels against the
    float64 oracle, the bars of test_gpu_raw).  Two views of different sizes
    in one call."""
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    K = np.array([[400.0, 0.0, shape[1] / 2], [0.0, 410.0, shape[0] / 2], [0.0, 0.0, 1.0]])
    M = np.eye(4)
    M[:3, :3] = [[0.8, 0.0, 0.6], [0.0, 1.0, 0.0], [-0.6, 0.0, 0.8]]
    M[:3, 3] = [0.1, -0.2, 0.3]
    views = [{"depth": _depth(*shape, 3), "K": K, "world_to_cam": M[:3]},
             {"depth": _depth(19, 70, 4), "K": K, "world_to_cam": M[:3]}]
    dev = [dict(v, depth=torch.from_numpy(v["depth"]).cuda()) for v in views]
    conf = [torch.full_like(v["depth"], -1.0) for v in dev]
    ctx = ftr.Context((64, 64, 64), np.array([-4, -4, -4, 4, 4, 4], np.float32))
    ctx.reset()
    ftr.ftr_splat_depth(ctx.h, dev, radius=radius, conf_out=conf)
    n = ctx.stats()[0]
    px = sum(v["depth"].size for v in views)
    buf = np.zeros(7 * px, np.float32)
    ftr.ftr_debug_buffer(ctx.h, 2, buf)
    ctx.close()
    P, N, W, maps = zip(*[oraw.raw_points(v["depth"], K, M[:3], radius=radius) for v in views])
    P, N, W = np.concatenate(P), np.concatenate(N), np.concatenate(W)
    assert n == len(P)
    assert np.abs(buf[:3 * n].reshape(-1, 3) - P).max(initial=0) <= 4e-6
    assert np.abs(buf[3 * px:3 * px + 3 * n].reshape(-1, 3) - N).max(initial=0) <= 1e-5
    assert np.abs(buf[6 * px:6 * px + n] - W).max(initial=0) <= 1e-5
    for a, b in zip(conf, maps):
        assert np.abs(a.cpu().numpy() - b).max() <= 1e-5
