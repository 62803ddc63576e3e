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
