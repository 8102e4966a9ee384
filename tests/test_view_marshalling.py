"""Camera matrices reach the C structs value by value in row-major order, from
every form a caller may hold them in; wrong sizes and dtypes are refused."""

import numpy as np
import pytest

from paper_1712_03084_gb300 import ftr

K = np.arange(9, dtype=np.float64).reshape(3, 3) + 0.1
RT = np.arange(12, dtype=np.float64).reshape(3, 4) - 0.3


@pytest.mark.parametrize("form", [
    lambda m: m, lambda m: m.astype(np.float32), lambda m: m.tolist(), lambda m: m.reshape(-1),
    lambda m: np.asfortranarray(m), lambda m: np.stack([m, m], -1)[..., 0], lambda m: m.astype(">f4"),
])
def test_matrices_in_every_form(form):
    d = np.ones((4, 5), np.float32)
    v = ftr.make_view(dict(depth=d, conf=d, rgb=np.zeros((6, 7, 3), np.uint8), K=form(K), world_to_cam=form(RT),
                           K_rgb=form(K), world_to_rgb=form(RT)))
    for got, want in ((v.K, K), (v.K_rgb, K), (v.world_to_cam, RT), (v.world_to_rgb, RT)):
        assert list(got) == [float(x) for x in want.astype(np.float32).reshape(-1)]
    assert (v.w, v.h, v.rgb_w, v.rgb_h) == (5, 4, 7, 6)
    cam = ftr.make_camera(form(K), form(RT), 8, 9)
    assert list(cam.K) == list(v.K) and list(cam.world_to_cam) == list(v.world_to_cam)


def test_wrong_sizes_and_dtypes_are_refused():
    torch = pytest.importorskip("torch")
    d = np.ones((4, 5), np.float32)
    with pytest.raises(ValueError):
        ftr.make_view(dict(depth=d, K=RT, world_to_cam=RT))
    with pytest.raises(ValueError):
        ftr.make_camera(K, K, 4, 5)
    with pytest.raises(TypeError):
        ftr.make_view(dict(depth=torch.ones(4, 5, dtype=torch.float64), K=K, world_to_cam=RT))
    with pytest.raises(TypeError):
        ftr.make_view(dict(depth=d.astype(np.float64), K=K, world_to_cam=RT))
    with pytest.raises(ValueError):
        ftr.make_view(dict(depth=torch.ones(5, 4).t(), K=K, world_to_cam=RT))
    t = torch.ones(4, 5)
    assert ftr.make_view(dict(depth=t, K=K, world_to_cam=RT)).depth == t.data_ptr()
