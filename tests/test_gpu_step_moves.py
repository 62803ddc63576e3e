"""The fused step's ways of moving master, m and v (16-byte copies shared by two lanes, 8-byte copies
per lane) and the compaction's forms (16-byte and element loads, several rounds per block).

The copies change no arithmetic, so a state whose planes are 16-byte aligned and the same state
8 bytes further (which takes the 8-byte copies) end the same but for the compiler's
contraction choices in the two kernels: a few ulps (2^-24 each) of the moments and of
the update, under 1e-6 relative L2 per plane. Index lists are integers and equal."""
import numpy as np
import pytest

from oracle import frustum as ofr
from paper_2606_09794_gb300 import inputs
from tests._parity import rel_l2

pytestmark = pytest.mark.gpu


def _at(x, offset):
    """x on the GPU, `offset` elements past a 256-byte boundary."""
    import torch
    x = torch.from_numpy(np.ascontiguousarray(x))
    buf = torch.empty(x.numel() + offset, dtype=x.dtype, device="cuda")
    buf[offset:] = x.reshape(-1).cuda()
    return buf[offset:].view(x.shape)


# lobes: slices of 2, 8 (two lanes idle), 16 (six idle) and 16 lanes; n so that the last warp is ragged
@pytest.mark.parametrize("n,L,frame,loss", [(1, 4, "quat", "given"), (513, 4, "cos", "mse"), (301, 12, "quat", "given"),
                                            (77, 20, "quat", "mse"), (4099, 8, "quat", "given"),
                                            (130, 32, "cos", "given")])
def test_copies_of_either_width_agree(lib, n, L, frame, loss):
    import torch
    w = inputs.point_cloud_workload(n, L, 300 + n + L, frame)
    rng = np.random.default_rng(n * L)
    m = (0.01 * rng.standard_normal(w.params.shape)).astype(np.float32)
    v = (1e-4 * (1 + rng.random(w.params.shape))).astype(np.float32)
    listed = np.flatnonzero(rng.random(n) < 0.6) if n > 1 else np.array([0])
    idx = np.concatenate([listed, [n, -1]]).astype(np.int32)  # entries outside [0, N) are skipped
    out = []
    for offset in (0, 2):
        st = lib.TrainState(_at(w.params, offset), _at(w.c0, 0), _at(m, offset), _at(v, offset))
        assert st.master.data_ptr() % 16 == 4 * offset
        rgb = torch.zeros((n, 3), device="cuda")
        lib.nasgabor_fused_step(st, _at(w.means, 0), w.cam, _at(w.g_rgb, 0), L, 3, idx=_at(idx, 0), frame_mode=frame,
                                rgb=rgb, loss=loss)
        lib.nasg_device_status()
        out.append([x.cpu().numpy() for x in (rgb, st.m, st.v, st.master)])
        lobes = (listed[:, None] * L + np.arange(L)).reshape(-1)
        hidden = np.setdiff1d(np.arange(n * L), lobes)
        np.testing.assert_array_equal(out[-1][3][:, hidden], w.params[:, hidden])
        np.testing.assert_array_equal(out[-1][1][:, hidden], m[:, hidden])
        assert (out[-1][3][:, lobes] != w.params[:, lobes]).mean() > 0.9
    (ra, ma, va, ta), (rb, mb, vb, tb) = out
    assert rel_l2(ra, rb) <= 1e-6
    for p in range(ma.shape[0]):
        assert rel_l2(ma[p], mb[p]) <= 1e-6 and rel_l2(va[p], vb[p]) <= 1e-6
        assert np.abs(ta[p] - tb[p]).max() <= 1e-6 * max(1.0, np.abs(tb[p]).max())


# one primitive, word and chunk edges, and more than 2048 chunks (two rounds per block)
@pytest.mark.parametrize("n", [1, 31, 33, 4096, 4099, 300_001, 2048 * 4096 + 4097])
def test_compaction_forms_agree(lib, n):
    import torch
    rng = np.random.default_rng(n)
    means = rng.uniform(-1.5, 1.5, (n, 3)).astype(np.float32)
    cam = inputs.shell_scene(2000, 1, 9, fov_sample=2000).cameras[2]
    lists = []
    for offset in (0, 1):
        idx, nv = lib.nasg_frustum_compact(_at(means, offset), cam.rot, cam.center, cam.tan_half_fov * 0.5)
        lists.append(idx[:int(nv.item())].cpu().numpy())
    np.testing.assert_array_equal(lists[0], lists[1])
    assert np.all(np.diff(lists[0]) > 0)
    ref = ofr.visible(means, cam.rot, cam.center, cam.tan_half_fov * 0.5)
    margin = ofr.boundary_margin(means, cam.rot, cam.center, cam.tan_half_fov * 0.5)
    got = np.zeros(n, bool)
    got[lists[0]] = True
    assert not ((got != ref) & (margin > 1e-5)).any()
