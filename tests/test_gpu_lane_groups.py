"""The register path with ceil(L/2) lanes per primitive (lobe counts whose slice would leave lanes
idle) against the staged path, over ragged numbers of primitives, lists with entries outside [0, N) and
both parameter types. An odd L is compared as the same mixture with one more lobe of weight 0 (raw
weight 0: tanh 0 = 0), which adds exactly 0 to every sum. The two paths sum the lobes of a primitive in
another order (at most 16 pairs, 2^-24 each): 2e-6 relative L2 per output plane."""
import pytest

pytestmark = pytest.mark.gpu


def _close(got, want, what):
    got, want = got.double(), want.double()
    assert float((got - want).norm()) <= 2e-6 * float(want.norm()), what


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("L,n", [(5, 8), (6, 1), (6, 4096), (9, 1000), (10, 333), (11, 2049), (12, 64), (17, 5), (18, 777),
                                 (19, 96), (20, 301)])
def test_groups_match_the_staged_path(lib, L, n, bf16):
    import torch
    from paper_2606_09794_gb300 import inputs
    dt = torch.bfloat16 if bf16 else torch.float32
    pad = (n + 7) // 8 * 8                       # the staged path's planes need whole 16-byte units
    full = L + L % 2
    sc = inputs.device_point_cloud(pad, full, 40 * L + n, "cuda", dt)
    if L % 2:
        sc["params"].view(10, pad, full)[7:10, :, -1] = 0
    args = (sc["c0"], sc["means"], sc["cam"], sc["g_rgb"])
    want = lib.nasgabor_fused_fwd_bwd(sc["params"], args[0], args[1], args[2], args[3], full)
    # the first n primitives by the register path: odd L or a list of them
    lobes = sc["params"].view(10, pad, full)[:, :n, :L]
    params, c0 = lobes.reshape(10, n * L).contiguous(), sc["c0"][:, :n].contiguous()
    means, g = sc["means"][:n].contiguous(), sc["g_rgb"][:n].contiguous()
    idx = torch.cat([torch.randperm(n, device="cuda"), torch.tensor([n, -1, n + 7], device="cuda")]).int()
    idx = idx[torch.randperm(n + 3, device="cuda")].contiguous()
    rgb = lib.nasgabor_eval_fwd(params, c0, means, sc["cam"], L, idx=idx)
    gp, gc, gm = lib.nasgabor_eval_bwd(params, means, sc["cam"], g, L, idx=idx)
    outs = [(rgb, gp, gc, gm)]
    if L % 2:
        outs.append(lib.nasgabor_fused_fwd_bwd(params, c0, means, sc["cam"], g, L))
    lib.nasg_device_status()
    wg = want[1].view(10, pad, full)[:, :n, :L].reshape(10, n * L)
    for r, p, c, m in outs:
        _close(r, want[0][:n], "rgb")
        _close(c, want[2][:, :n], "c0")
        _close(m, want[3][:n], "means")
        for k in range(10):
            _close(p[k], wg[k], k)
