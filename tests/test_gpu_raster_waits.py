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
