"""The batched launch with three items per thread and sub-tile (BF16 batches of many sub-tiles)
against the single-scene fused pass, over scenes whose last sub-tiles are ragged, whose lobe counts
take each arithmetic instance, and which are staged and loaded directly; and the same scenes few enough
for two items. Both evaluate the same formulas in FP32 with FP32 sums over at most 16 lanes; the
instances differ in summation order and contraction (a few 2^-24 per operation): 2e-6 relative L2 per
output."""
import pytest


pytestmark = pytest.mark.gpu


# sizes: about 2.6e6 lanes (three items) and 6e4 (two); L = 6 and 5 (general instances), 2 (direct
# loads only), 4, 8, 16 (fixed instances)
@pytest.mark.parametrize("scale", [1.0, 0.02])
@pytest.mark.parametrize("staged,dynamic,sub_tiles", [(1, 1, 2), (1, 0, 1), (0, 1, 4)])
@pytest.mark.parametrize("lobes", [(8, 16, 4), (8, 6, 2, 16), (8, 5, 16)])
def test_batch_matches_single_scenes(lib, scale, staged, dynamic, sub_tiles, lobes):
    import torch
    from paper_2606_09794_gb300 import inputs
    sizes = {8: 400_003, 16: 120_001, 4: 50_000, 6: 77_777, 2: 60_001, 5: 70_001}
    scenes = []
    for j, L in enumerate(lobes):
        n = max(1, int(sizes[L] * scale))
        sc = inputs.device_point_cloud(n, L, 900 + j, "cuda", torch.bfloat16)
        scenes.append(sc)
    b = lib.Batch(scenes, sub_tiles=sub_tiles)
    b.tuning.staged, b.tuning.dynamic = staged, dynamic
    b.run()
    lib.nasg_device_status()
    for sc in scenes:
        ref = lib.nasgabor_fused_fwd_bwd(sc["params"], sc["c0"], sc["means"], sc["cam"], sc["g_rgb"], sc["n_lobes"])
        for name, r in zip(("rgb", "g_params", "g_c0", "g_means"), ref):
            got, want = sc[name].double(), r.double()
            assert bool(torch.isfinite(got).all())
            rows = got.shape[0] if name in ("g_params", "g_c0") else 1
            for k in range(rows):
                g, w = (got[k], want[k]) if rows > 1 else (got, want)
                assert float((g - w).norm()) <= 2e-6 * float(w.norm()), (name, k, sc["n_lobes"])
