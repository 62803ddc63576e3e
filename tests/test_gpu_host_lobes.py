"""The fused pass on page-locked host arrays at lobe counts that leave lanes of a slice idle, against the
device-resident pass, which gives such a primitive fewer lanes: other orders of the same FP32 sums over at most 16
lanes, 2e-6 relative L2 per output plane as tests/test_gpu_lane_groups.py states it."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n", [(5, 1003), (6, 77), (9, 333), (12, 64), (17, 5), (20, 301)])
@pytest.mark.parametrize("bf16", [False, True])
def test_host_arrays(lib, L, n, bf16):
    import torch
    from paper_2606_09794_gb300 import inputs
    sc = inputs.device_point_cloud(n, L, 11 * L + n, "cuda", torch.bfloat16 if bf16 else torch.float32)
    names = ("params", "c0", "means", "g_rgb")
    ref = lib.nasgabor_fused_fwd_bwd(sc["params"], sc["c0"], sc["means"], sc["cam"], sc["g_rgb"], L)
    p, c0, mu, g = [sc[k].cpu().pin_memory() for k in names]
    out = tuple(torch.full(t.shape, float("nan")).pin_memory() for t in ref)
    lib.HostFused(n, L, p.dtype)(p, c0, mu, sc["cam"], g, out)
    torch.cuda.synchronize()
    for j, (got, want) in enumerate(zip(out, ref)):
        rows = range(got.shape[0]) if j in (1, 2) else [slice(None)]
        for k in rows:
            x, y = got[k].double(), want[k].double().cpu()
            assert float((x - y).norm()) <= 2e-6 * float(y.norm()), (j, k)
