"""How a compositing call waits, and what it leaves behind when it ends without an image."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _scene(n, seed, scale):
    """Centres in the cube [-1, 1]^3, all in front of the camera of _camera."""
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rand = lambda *shape: torch.rand(shape, generator=gen, device="cuda")
    quats = torch.randn((n, 4), generator=gen, device="cuda")
    return rand(n, 3) * 2.0 - 1.0, rand(n, 3) * scale + 0.5 * scale, quats, rand(n) * 0.9 + 0.05, rand(n, 3)


def _camera(lib, w, h):
    return lib.raster_camera(np.eye(3), (0.0, 0.0, -4.0), w, h, 0.5 * w / 0.4)


def test_refused_forward_leaves_nothing_running(lib):
    """2^22 primitives, room for 16 pairs, on a side stream: the call returns its status with the stream
    idle (the depth sort of so many takes a few hundred microseconds after the count is known)."""
    import torch
    n = 1 << 22
    args = _scene(n, 5, 1e-3)
    r = lib.Raster(n, _camera(lib, 320, 180), 16)
    image, T = torch.empty((180, 320, 3), device="cuda"), torch.empty((180, 320), device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        with pytest.raises(lib.NasgError) as e:
            r.forward(*args, image=image, final_t=T, stream=side)
        idle = side.query()
        assert e.value.status == -7
        assert idle


# The host waits 0.2 s for the work in front of the projection. With the context's blocking-sync flag the
# thread sleeps meanwhile (a spinning one would spend all of the wait on its core).
BLOCKING = """
import ctypes, sys, time
sys.path.insert(0, {root!r})
cuda = ctypes.CDLL("libcuda.so.1")
assert cuda.cuInit(0) == 0 and cuda.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0  # CU_CTX_SCHED_BLOCKING_SYNC
import torch
from paper_2606_09794_gb300 import binding as lib
from tests.test_gpu_raster_waits import _camera, _scene
args = _scene(1000, 3, 0.01)
r = lib.Raster(1000, _camera(lib, 64, 48), 1 << 16)
want = r.forward(*args)[0].clone()
flags, active = ctypes.c_uint(), ctypes.c_int()
assert cuda.cuDevicePrimaryCtxGetState(0, ctypes.byref(flags), ctypes.byref(active)) == 0 and flags.value & 7 == 4
torch.cuda.synchronize()
torch.cuda._sleep(400_000_000)
t, c = time.monotonic(), time.thread_time()
got = r.forward(*args)[0]
t, c = time.monotonic() - t, time.thread_time() - c
assert torch.equal(got, want)
assert t > 0.1, t
assert c < 0.5 * t, (c, t)
"""


def test_forward_waits_blocked_where_the_device_asks_for_it(lib):
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    res = subprocess.run([sys.executable, "-c", BLOCKING.format(root=root)], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]


def test_look_back_gives_up(lib):
    """Blocks whose first predecessor never publishes its counts: every one gives up, says so to those after
    it, in the failure word and in the device status. With that predecessor they place all their entries."""
    lib.nasg_device_status()
    placed, before, failed = lib.nasg_probe_look_back_timeout(1 << 20, first=0)
    lib.nasg_device_status()
    assert placed == [1024] * lib.LOOK_BACK_BLOCKS and before == list(range(1, lib.LOOK_BACK_BLOCKS + 1)) and failed == 0
    placed, before, failed = lib.nasg_probe_look_back_timeout(1024, first=1)
    assert placed == [-1] * lib.LOOK_BACK_BLOCKS and before == [-1] * lib.LOOK_BACK_BLOCKS and failed == 1
    with pytest.raises(lib.NasgError) as e:
        lib.nasg_device_status()
    assert e.value.status == -6
    lib.nasg_device_status()


# 20 x 12 tiles (one pixel per lane) and 60 x 34 (two); small and large sort blocks
@pytest.mark.parametrize("where", [1, 2])
@pytest.mark.parametrize("w,h,n,scale", [(320, 192, 5000, 0.05), (960, 540, 450_000, 0.01)])
def test_failed_lists_give_an_empty_image(lib, where, w, h, n, scale):
    import ctypes

    import torch
    args = _scene(n, 8, scale)
    r = lib.Raster(n, _camera(lib, w, h), 1 << 25)
    want, T = r.forward(*args)
    g = torch.randn((h, w, 3), device="cuda")
    ref = r.backward(args[4], T, g)
    assert float(T.min()) < 0.9 and float(ref[1].abs().max()) > 0
    image, final_t = torch.full((h, w, 3), 7.0, device="cuda"), torch.full((h, w), 7.0, device="cuda")
    p = [lib._ptr(t) for t in args]
    lib._check(lib.lib.nasg_probe_raster_failed(where, n, *p, ctypes.byref(r.camera), lib._ptr(image), lib._ptr(final_t),
                                                r.max_pairs, lib._ptr(r.workspace), r.workspace.numel(), lib._stream(None)),
               "nasg_probe_raster_failed")
    assert float(image.abs().max()) == 0.0 and float(final_t.min()) == 1.0 and float(final_t.max()) == 1.0
    gc, go = r.backward(args[4], final_t, g)
    assert float(gc.abs().max()) == 0.0 and float(go.abs().max()) == 0.0
    lib.nasg_device_status()
    again, _ = r.forward(*args)  # the next forward starts afresh
    assert torch.equal(again, want)


# room for the first image's pairs (at most 4 and 64 tiles each), not for every primitive in all 12 and 1200 tiles
@pytest.mark.parametrize("w,h,room", [(64, 48, 8000), (640, 480, 128_000)])
def test_backward_after_a_refused_forward(lib, w, h, room):
    """The refused forward leaves its workspace the counts of the image before it and no lists: gradients zero."""
    import torch
    n = 2000
    args = _scene(n, 9, 0.03)
    r = lib.Raster(n, _camera(lib, w, h), room)
    _, T = r.forward(*args)
    g = torch.randn((h, w, 3), device="cuda")
    assert float(r.backward(args[4], T, g)[1].abs().max()) > 0
    with pytest.raises(lib.NasgError) as e:
        r.forward(args[0], args[1] * 1e4, *args[2:])
    assert e.value.status == -7
    gc, go = r.backward(args[4], T, g)
    assert float(gc.abs().max()) == 0.0 and float(go.abs().max()) == 0.0
