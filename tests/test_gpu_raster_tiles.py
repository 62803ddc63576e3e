"""The rendering kernels' two pixel layouts (two pixels per lane for images of many tiles, one
for few) and their sub-tile lists against the FP64 oracle, in a window of the image that starts
and ends inside tiles. The oracle renders the window as an image of its own whose principal point
is shifted by the window's corner. Bounds as tests/test_gpu_raster.py states them: FP32 colours
within 5e-5, gradients within 1e-4 relative L2, decisions within 1e-4 of a threshold excluded."""
import numpy as np
import pytest

from oracle import raster as orr
from tests._parity import rel_l2

pytestmark = pytest.mark.gpu

MARGIN = 1e-4


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()


# (width, height, window corner and size, primitives, log-scale range): 27 x 26 = 702 and 700 x 1
# tiles run two pixels per lane, the others one; the last list holds several staged batches
@pytest.mark.parametrize("w,h,win,n,log_scale", [
    (432, 416, (201, 190, 33, 22), 300, (-4.5, -1.5)),
    (11193, 9, (5590, 0, 40, 9), 250, (-3.0, -1.5)),
    (37, 21, (0, 0, 37, 21), 300, (-4.5, -1.5)),
    (17, 1, (0, 0, 17, 1), 60, (-3.0, -1.0)),
    (48, 33, (9, 5, 30, 28), 1500, (-4.0, -2.0)),
])
def test_window_matches_oracle(lib, w, h, win, n, log_scale):
    import torch
    rng = np.random.default_rng(w + 7 * n)
    sc = [rng.uniform(-1, 1, (n, 3)), np.exp(rng.uniform(*log_scale, (n, 3))), rng.normal(size=(n, 4)),
          rng.uniform(0.003, 0.98, n), rng.uniform(0, 1, (n, 3))]
    sc = [x.astype(np.float32) for x in sc]
    centre, fx = (0.0, 0.0, -4.0), np.float32(0.5 * max(w if w < 1000 else 400, h) / 0.4)
    cam = lib.raster_camera(np.eye(3), centre, w, h, fx)
    r = lib.Raster(n, cam, 1 << 22)
    dev = [_dev(x) for x in sc]
    img, T = r.forward(*dev)
    x0, y0, ww, wh = win
    ocam = {"rot": np.eye(3), "centre": np.asarray(centre), "fx": fx, "fy": fx, "cx": 0.5 * w - x0,
            "cy": 0.5 * h - y0, "near": np.float32(0.2)}
    ref, tref, margin = orr.render(*sc, ocam, ww, wh, with_margin=True)
    ok = margin > MARGIN
    assert ok.mean() > 0.9, ok.mean()
    cut = (slice(y0, y0 + wh), slice(x0, x0 + ww))
    assert np.abs(img.cpu().numpy()[cut] - ref)[ok].max() <= 5e-5
    assert np.abs(T.cpu().numpy()[cut] - tref)[ok].max() <= 5e-5
    g = rng.normal(size=(wh, ww, 3))
    g[~ok] = 0.0
    full = np.zeros((h, w, 3))
    full[cut] = g
    gc, go = r.backward(dev[4], T, _dev(full))
    torch.cuda.synchronize()
    rc, ro = orr.render_backward(*sc, ocam, ww, wh, g)
    assert np.abs(rc).max() > 0
    assert rel_l2(gc.cpu().numpy(), rc) <= 1e-4
    assert rel_l2(go.cpu().numpy(), ro) <= 1e-4
