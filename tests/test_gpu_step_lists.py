"""The fused step by index lists at four lobes, where each warp chooses its copies by whether its 16 entries are
neighbours: runs, gaps, any order, entries outside [0, N) inside a warp and a ragged last warp; and L = 12. Against
the same state 8 bytes further, whose planes allow the 8-byte copies only. The copies change no arithmetic:
under 1e-6 relative L2 per plane for the kernels' contraction choices, as tests/test_gpu_step_moves.py states it."""
import numpy as np
import pytest

from paper_2606_09794_gb300 import inputs
from tests._parity import rel_l2
from tests.test_gpu_step_moves import _at

pytestmark = pytest.mark.gpu

N = 3001


def _lists():
    rng = np.random.default_rng(4)
    some = np.flatnonzero(rng.random(N) < 0.45)
    runs = np.concatenate([np.arange(a, a + 16 + a % 37) for a in range(0, N - 60, 100)])
    skipped = runs.copy()
    skipped[5::16] = -1
    skipped[7::48] = N
    return {"all": np.arange(N), "runs": runs, "from_17": np.arange(17, 17 + 16 * 9 + 5), "gaps": some,
            "any_order": rng.permutation(some), "downward": np.arange(N - 1, 100, -1), "skipped": skipped, "one": np.array([N - 1])}


@pytest.mark.parametrize("name", sorted(_lists()))
@pytest.mark.parametrize("L", [4, 12])
def test_lists(lib, L, name):
    import torch
    entries = _lists()[name].astype(np.int32)
    w = inputs.point_cloud_workload(N, L, 70 + L, "quat")
    rng = np.random.default_rng(L)
    m = (0.01 * rng.standard_normal(w.params.shape)).astype(np.float32)
    v = (1e-4 * (1 + rng.random(w.params.shape))).astype(np.float32)
    out = []
    for offset in (0, 2):
        st = lib.TrainState(_at(w.params, offset), _at(w.c0, 0), _at(m, offset), _at(v, offset))
        rgb = torch.zeros((N, 3), device="cuda")
        lib.nasgabor_fused_step(st, _at(w.means, 0), w.cam, _at(w.g_rgb, 0), L, 3, idx=_at(entries, 0), rgb=rgb)
        lib.nasg_device_status()
        out.append([x.cpu().numpy() for x in (rgb, st.m, st.v, st.master)])
    listed = np.unique(entries[(entries >= 0) & (entries < N)])
    lobes = (listed[:, None] * L + np.arange(L)).reshape(-1)
    hidden = np.setdiff1d(np.arange(N * L), lobes)
    (ra, ma, va, ta), (rb, mb, vb, tb) = out
    np.testing.assert_array_equal(ta[:, hidden], w.params[:, hidden])
    np.testing.assert_array_equal(ma[:, hidden], m[:, hidden])
    assert (ta[:, lobes] != w.params[:, lobes]).mean() > 0.9
    assert rel_l2(ra, rb) <= 1e-6
    for p in range(ma.shape[0]):
        assert rel_l2(ma[p], mb[p]) <= 1e-6 and rel_l2(va[p], vb[p]) <= 1e-6
        assert np.abs(ta[p] - tb[p]).max() <= 1e-6 * max(1.0, np.abs(tb[p]).max())
