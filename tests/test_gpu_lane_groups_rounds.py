"""The register path either side of the line between slices and groups of ceil(L/2) lanes (whether the groups save
a round of the persistent grid), against the staged path over the same primitives; as
tests/test_gpu_lane_groups.py: an odd L compared as the same mixture with one more lobe of weight 0, list entries
outside [0, N) skipped, 2e-6 relative L2 per output plane."""
import pytest

pytestmark = pytest.mark.gpu


def _close(got, want, what):
    got, want = got.double(), want.double()
    assert float((got - want).norm()) <= 2e-6 * float(want.norm()), what


# many rounds; just over one round of slices at two and at three blocks per SM (152 x 512 and 152 x 768 lanes)
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("L,n", [(5, 120_007), (5, 19_457), (6, 120_007), (9, 60_001), (9, 9_729), (10, 60_001), (11, 14_593),
                                 (12, 60_001), (17, 40_003), (17, 4_865), (18, 7_297), (19, 40_003), (20, 40_003)])
def test_either_side_of_the_line(lib, L, n, bf16):
    import torch
    from paper_2606_09794_gb300 import inputs
    dt = torch.bfloat16 if bf16 else torch.float32
    pad = (n + 7) // 8 * 8                       # the staged path's planes need whole 16-byte units
    full = L + L % 2
    sc = inputs.device_point_cloud(pad, full, 50 * L + n, "cuda", dt)
    if L % 2:
        sc["params"].view(10, pad, full)[7:10, :, -1] = 0
    cam = sc["cam"]
    want = lib.nasgabor_fused_fwd_bwd(sc["params"], sc["c0"], sc["means"], cam, sc["g_rgb"], full)
    params = sc["params"].view(10, pad, full)[:, :, :L].reshape(10, pad * L).contiguous()
    g_want = want[1].view(10, pad, full)[:, :, :L].reshape(10, pad * L)
    idx = torch.arange(n, device="cuda", dtype=torch.int32)
    listed = torch.cat([idx, torch.tensor([-1, pad, 2 ** 31 - 1], device="cuda", dtype=torch.int32)])
    rgb, gp = torch.zeros((pad, 3), device="cuda"), torch.zeros((10, pad * L), device="cuda")
    gc, gm = torch.zeros((3, pad), device="cuda"), torch.zeros((pad, 3), device="cuda")
    lib.nasgabor_eval_fwd(params, sc["c0"], sc["means"], cam, L, idx=listed, rgb=rgb)
    lib.nasgabor_eval_bwd(params, sc["means"], cam, sc["g_rgb"], L, idx=listed, g_params=gp, g_c0=gc, g_means=gm)
    lib.nasg_device_status()
    assert not rgb[n:].any() and not gp[:, n * L:].any() and not gc[:, n:].any() and not gm[n:].any()
    _close(rgb[:n], want[0][:n], "rgb")
    _close(gm[:n], want[3][:n], "g_means")
    for k in range(10):
        _close(gp[k, :n * L], g_want[k, :n * L], ("g_params", k))
    for k in range(3):
        _close(gc[k, :n], want[2][k, :n], ("g_c0", k))
    if L % 2:                                    # odd lobe counts take this path without a list too
        one = lib.nasgabor_fused_fwd_bwd(params, sc["c0"], sc["means"], cam, sc["g_rgb"], L)
        _close(one[0], want[0], "fused rgb")
        _close(one[3], want[3], "fused g_means")
        for k in range(10):
            _close(one[1][k], g_want[k], ("fused g_params", k))
