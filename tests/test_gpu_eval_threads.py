"""Contexts on several host threads evaluate images of different heights: the
column pass needs more than 48 KB of shared memory above 6144 rows, an amount
that is set per function and device, not per context.  Every call gives what the
same call gives alone."""

import threading

import numpy as np
import pytest

from tests import gpu_common as G

pytestmark = pytest.mark.gpu


def test_tall_images_on_several_threads():
    torch = G.require_gpu()
    from paper_1712_03084_gb300 import ftr
    K = np.array([[400.0, 0, 2], [0, 400.0, 3000], [0, 0, 1]], np.float32)
    RT = np.eye(3, 4, dtype=np.float32)
    jobs = []
    for h in (6200, 16384, 6200, 16384):
        rng = np.random.default_rng(h)
        depth = [torch.from_numpy(np.where(rng.random((h, 4)) < 0.001, 1.5, 0.0).astype(np.float32)).cuda()
                 for _ in range(2)]
        ctx = ftr.Context((64, 64, 64), (-1, -1, -1, 1, 1, 1))
        cam = ftr.make_camera(K, RT, 4, h)
        jobs.append((ctx, cam, depth, ftr.ftr_eval_geometry(ctx.h, cam, *depth)))
    torch.cuda.synchronize()
    wrong = []

    def work(ctx, cam, depth, want):
        try:
            for _ in range(1500):
                if ftr.ftr_eval_geometry(ctx.h, cam, *depth) != want:
                    wrong.append("result")
        except Exception as e:                           # reported by the main thread
            wrong.append(repr(e))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for j in jobs:
        j[0].close()
    assert not wrong, wrong[:3]
