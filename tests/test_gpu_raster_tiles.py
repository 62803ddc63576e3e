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
# tiles run two pixels per lane in the backward, 37 x 33 = 1221 in the forward too, the others one;
# the last list holds several staged batches
@pytest.mark.parametrize("w,h,win,n,log_scale", [
    (432, 416, (201, 190, 33, 22), 300, (-4.5, -1.5)),
    (592, 521, (281, 243, 33, 22), 300, (-4.5, -1.5)),
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


# The binning at the edges of its forms: one tile, 256 tiles (a single-digit tile key), keys of three
# and four digits (over 256 tile columns or rows), lists shorter and longer than a sort block of
# either shape, primitives that span more tiles than a thread lists alone, depths that tie by the
# hundred (order by index), nothing but ties, and more primitives than the small depth blocks take.
@pytest.mark.parametrize("w,h,n,log_scale,depths", [
    (16, 16, 40, (-3.0, -1.5), 0),
    (256, 256, 900, (-3.5, -1.0), 3),
    (4200, 40, 1100, (-4.0, -0.5), 0),
    (24, 4200, 1100, (-4.0, -0.5), 5),
    (4500, 4300, 700, (-3.5, -0.3), 2),
    (640, 360, 4096, (-4.5, -2.5), 1),
    (1280, 720, 20_000, (-4.5, -2.0), 40),
    (640, 360, 450_000, (-6.5, -4.0), 1000),
])
def test_binning_forms(lib, w, h, n, log_scale, depths):
    import torch
    rng = np.random.default_rng(w + h + n)
    half = np.array([1.0, 1.0 * h / w]) if w >= h else np.array([1.0 * w / h, 1.0])
    means = np.concatenate([rng.uniform(-1.1, 1.1, (n, 2)) * half, rng.uniform(-1, 1, (n, 1))], axis=1)
    if depths:
        means[:, 2] = rng.integers(0, depths, n) * (1.0 / depths) - 0.5
    sc = [means, np.exp(rng.uniform(*log_scale, (n, 3))) * half.min() ** 0.5, rng.normal(size=(n, 4)),
          rng.uniform(0.01, 0.9, n), rng.uniform(0, 1, (n, 3))]
    sc = [x.astype(np.float32) for x in sc]
    fx = np.float32(max(w, h) / 0.5)
    centre = (0.0, 0.0, -4.0)
    cam = lib.raster_camera(np.eye(3), centre, w, h, fx)
    r = lib.Raster(n, cam, 1 << 26)
    img, T = r.forward(*[_dev(x) for x in sc])
    lib.nasg_device_status()
    pix = np.stack([rng.integers(0, w, 60), rng.integers(0, h, 60)], axis=1)
    ocam = {"rot": np.eye(3), "centre": np.asarray(centre), "fx": fx, "fy": fx, "cx": 0.5 * w, "cy": 0.5 * h,
            "near": np.float32(0.2)}
    ref, tref, margin = orr.render(*sc, ocam, w, h, pixels=pix, with_margin=True)
    ok = margin > MARGIN
    assert ok.mean() > 0.7, ok.mean()
    assert (tref < 1).any()
    assert np.abs(img.cpu().numpy()[pix[:, 1], pix[:, 0]] - ref)[ok].max() <= 1e-4
    assert np.abs(T.cpu().numpy()[pix[:, 1], pix[:, 0]] - tref)[ok].max() <= 1e-4
    # lists that differ in order would differ in the image; a second run gives the same bits
    again, _ = r.forward(*[_dev(x) for x in sc])
    torch.testing.assert_close(again, img, rtol=0, atol=0)


def _frame(lib, n, w, h, seed):
    rng = np.random.default_rng(seed)
    sc = [rng.uniform(-1, 1, (n, 3)), np.exp(rng.uniform(-4.0, -1.8, (n, 3))), rng.normal(size=(n, 4)),
          rng.uniform(0.02, 0.98, n), rng.uniform(0, 1, (n, 3))]
    sc = [x.astype(np.float32) for x in sc]
    fx = np.float32(0.5 * max(w, h) / 0.4)
    cam = lib.raster_camera(np.eye(3), (0.0, 0.0, -4.0), w, h, fx)
    ocam = {"rot": np.eye(3), "centre": np.array([0.0, 0.0, -4.0]), "fx": fx, "fy": fx, "cx": 0.5 * w, "cy": 0.5 * h,
            "near": np.float32(0.2)}
    r = lib.Raster(n, cam, 1 << 23)
    dev = [_dev(x) for x in sc]
    img, T = r.forward(*dev)
    return r, sc, dev, T, ocam, rng


# an infinite or NaN upstream gradient at one pixel reaches the primitives that contribute there, an
# infinite colour those in front of it at the pixels it contributes to, and no others
@pytest.mark.parametrize("w,h,n", [(432, 416, 1500), (40, 16, 200)])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_backward_keeps_non_finite_values_where_they_are(lib, w, h, n, bad):
    r, sc, dev, T, ocam, rng = _frame(lib, n, w, h, 78)
    g = rng.normal(size=(h, w, 3)).astype(np.float32)
    px, py = w // 2 + 3, h // 2 - 2
    ref_c, ref_o = (x.cpu().numpy() for x in r.backward(dev[4], T, _dev(g)))
    g[py, px] = bad
    gc, go = (x.cpu().numpy() for x in r.backward(dev[4], T, _dev(g)))
    z, mean2, sigma2, valid = orr.project(*sc[:3], ocam)
    alpha, _ = orr._alphas(px + 0.5, py + 0.5, mean2, sigma2, sc[3])
    may = valid & (alpha >= (1 - MARGIN) * orr.ALPHA_MIN)   # all that could contribute at the pixel
    touched = ~np.isfinite(gc).all(1)
    assert touched.any() and not (touched & ~may).any()
    assert not ((~np.isfinite(go)) & ~may).any()
    assert rel_l2(gc[~may], ref_c[~may]) <= 1e-5 and rel_l2(go[~may], ref_o[~may]) <= 1e-5


def test_refused_forward_stays_inside_its_workspace(lib):
    """64 primitives over 65,536 tiles each, room for 16 pairs: the call is refused, the pair count
    reported, and nothing past the workspace's end written, where the tables of 4.2e6 pairs would lie."""
    import torch
    n, w, h = 64, 4096, 4096
    cam = lib.raster_camera(np.eye(3), (0.0, 0.0, -4.0), w, h, 5000.0)
    r = lib.Raster(n, cam, 16)
    nbytes = r.workspace.numel()
    buf = torch.full((nbytes + (1 << 22),), 0xA5, dtype=torch.uint8, device="cuda")
    r.workspace = buf[:nbytes]
    means = torch.zeros((n, 3), device="cuda")
    scales = torch.full((n, 3), 50.0, device="cuda")
    quats = torch.tensor([[1.0, 0.0, 0.0, 0.0]], device="cuda").repeat(n, 1)
    image = torch.full((h, w, 3), 7.0, device="cuda")
    with pytest.raises(lib.NasgError) as e:
        r.forward(means, scales, quats, torch.full((n,), 0.5, device="cuda"), torch.ones((n, 3), device="cuda"), image=image)
    assert e.value.status == -7
    torch.cuda.synchronize()
    assert bool((buf[nbytes:] == 0xA5).all())
    assert bool((image == 7.0).all())


def test_forward_under_capture(lib):
    """Without primitives a forward needs no wait and can be captured."""
    import torch
    cam = lib.raster_camera(np.eye(3), (0.0, 0.0, -4.0), 40, 24, 50.0)
    empty = lib.Raster(0, cam, 16)
    e3, image, T = torch.empty((0, 3), device="cuda"), torch.ones((24, 40, 3), device="cuda"), torch.zeros((24, 40), device="cuda")
    args = (e3, e3, torch.empty((0, 4), device="cuda"), torch.empty(0, device="cuda"), e3)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        empty.forward(*args, image=image, final_t=T)
    graph.replay()
    torch.cuda.synchronize()
    assert float(image.abs().max()) == 0.0 and float(T.min()) == 1.0


def test_forward_beside_a_capture(lib):
    """A forward on another thread and stream, its first there, while this thread captures: neither
    it nor that thread's end disturbs the capture."""
    import threading

    import torch
    rng = np.random.default_rng(11)
    n = 50
    args = [_dev(x) for x in (rng.uniform(-1, 1, (n, 3)), np.full((n, 3), 0.05), rng.normal(size=(n, 4)),
                              np.full(n, 0.5), rng.uniform(size=(n, 3)))]
    cam = lib.raster_camera(np.eye(3), (0.0, 0.0, -4.0), 40, 24, 50.0)
    want = lib.Raster(n, cam, 1 << 12).forward(*args)[0].clone()
    beside, other = lib.Raster(n, cam, 1 << 12), torch.cuda.Stream()
    image, T, x = torch.empty_like(want), torch.empty((24, 40), device="cuda"), torch.zeros(8, device="cuda")
    errors = []

    def run():
        try:
            beside.forward(*args, image=image, final_t=T, stream=other)
        except Exception as e:  # reported below, after the capture has ended
            errors.append(e)

    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        x.add_(1.0)
        thread = threading.Thread(target=run)
        thread.start()
        thread.join()
        x.add_(1.0)
    graph.replay()
    torch.cuda.synchronize()
    assert not errors
    assert torch.equal(image, want) and float(x.sum()) == 16.0
