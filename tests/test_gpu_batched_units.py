"""The batched launch's two divisions of the work (tiles of the direct kernel, sub-tiles of the staged one)
over scenes that end inside either, hold one primitive or none, first, between and last. Every schedule runs
the same arithmetic on each primitive, so all give the same bits; and the BF16 batch agrees with the
single-scene fused pass within the 2e-6 relative L2 per output of tests/test_gpu_batched_items.py."""
import pytest

pytestmark = pytest.mark.gpu

# (primitives, lobes) of the scenes: few sub-tiles; three items per thread; most of the lanes with odd lobe counts
FEW = [(0, 8), (1, 8), (127, 4), (0, 4), (129, 16), (700, 6), (385, 8), (0, 16)]
MANY = [(0, 8), (400_003, 8), (1, 4), (50_001, 4), (0, 16), (30_000, 16), (191, 8), (0, 8)]
ODD = [(300_001, 5), (1, 3), (0, 5), (90_001, 9), (20_000, 8), (0, 3)]


OUTPUTS = ("rgb", "g_params", "g_c0", "g_means")


def _scenes(sizes, dtype):
    from paper_2606_09794_gb300 import inputs
    scenes = []
    for j, (n, L) in enumerate(sizes):
        sc = inputs.device_point_cloud(max(n, 1), L, 300 + j, "cuda", dtype)
        if n == 0:
            sc.update(params=sc["params"][:, :0].contiguous(), c0=sc["c0"][:, :0].contiguous(), means=sc["means"][:0],
                      g_rgb=sc["g_rgb"][:0])
        scenes.append(sc)
    return scenes


def _run(lib, scenes, staged, dynamic, sub_tiles):
    b = lib.Batch(scenes, sub_tiles=sub_tiles)
    b.tuning.staged, b.tuning.dynamic = staged, dynamic
    for sc in scenes:
        for name in OUTPUTS:
            sc[name].fill_(float("nan"))
    b.run()
    lib.nasg_device_status()
    return [[sc[name] for name in OUTPUTS] for sc in scenes]  # each Batch allocates its own


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("sizes", [FEW, MANY, ODD], ids=["few", "many", "odd"])
def test_schedules_agree(lib, sizes, dtype):
    import torch
    scenes = _scenes(sizes, torch.bfloat16 if dtype == "bf16" else torch.float32)
    want = _run(lib, scenes, 0, 0, 1)
    assert all(bool(torch.isfinite(t).all()) for outs in want for t in outs)
    for staged, dynamic, sub_tiles in ((0, 1, 1), (0, 0, 3), (0, 1, 64), (1, 1, 1), (1, 0, 3), (1, 1, 64)):
        got = _run(lib, scenes, staged, dynamic, sub_tiles)
        for g, w in zip(got, want):
            for x, y in zip(g, w):
                assert torch.equal(x, y), (staged, dynamic, sub_tiles)


@pytest.mark.parametrize("sizes", [FEW, MANY, ODD], ids=["few", "many", "odd"])
def test_batch_matches_single_scenes(lib, sizes):
    import torch
    scenes = _scenes(sizes, torch.bfloat16)
    for sc, outs in zip(scenes, _run(lib, scenes, 1, 1, 2)):
        if sc["means"].shape[0] == 0:
            continue
        ref = lib.nasgabor_fused_fwd_bwd(sc["params"], sc["c0"], sc["means"], sc["cam"], sc["g_rgb"], sc["n_lobes"])
        for name, got, want in zip(OUTPUTS, outs, ref):
            assert float((got.double() - want.double()).norm()) <= 2e-6 * float(want.double().norm()), (name, sc["n_lobes"])
