"""Timed cases of the NASGabor appearance library, over its public entry points.

Each case is one call, or the few calls that belong together, of a program that uses the
library: colours for a viewer, forward and backward for an optimiser, the fused training and
fitting steps, the batched launch over many scenes, compositing, and a whole training frame.
Inputs are drawn on the GPU from the seed alone, with the distributions of the library's
synthetic workloads (paper_2606_09794_gb300/inputs.py): log-uniform sharpness in [1, 1e3],
anisotropy in [0, 1], carrier frequency in [0, 8], weights in [0, 1].

`exact` restates every path in 64-bit torch, apart from the library's code: the lobe by its
definition (gradients by torch autograd), real spherical harmonics from associated Legendre
polynomials, Adam as torch.optim.Adam writes it, and compositing by cumulative products over
each tile's primitives in depth order.
"""
import math

import torch

from paper_2606_09794_gb300 import binding as nb

DEV = "cuda"
CENTRE_CLOUD = (0.0, 0.0, 3.0)    # the point clouds' camera
CENTRE_FRAME = (0.0, 0.0, -4.0)   # the compositing camera, looking along +z
FRAME_TAN = 0.6                   # its horizontal half field of view
ADAM = dict(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8)
FIRST_STEP = 100                  # training states are met in mid-training (m, v not zero)
PAIR_CAP = 1 << 26                # room for (tile, primitive) pairs of a frame
FIELDS = {"nasgabor": ("lam", "a", "k"), "nasg": ("lam", "a"), "sg": ("lam",), "phase": ("lam", "a", "k", "phi")}


def listed():
    return [
        # The smallest call: a few thousand primitives coloured for a preview or a unit of a larger
        # program. Launch and call overhead count.
        {"name": "colours_4k", "kind": "eval", "mode": "forward", "n": 4096, "lobes": 4, "dtype": "f32",
         "frame": "quat", "norm": "approx", "family": "nasgabor"},
        # An optimiser step's appearance part written in PyTorch: NasgEval.apply(...).backward(g).
        {"name": "autograd_f32_1m", "kind": "eval", "mode": "autograd", "n": 1_000_000, "lobes": 8, "dtype": "f32",
         "frame": "quat", "norm": "approx", "family": "nasgabor"},
        # The same size as one fused pass over BF16-stored parameters.
        {"name": "fused_bf16_1m", "kind": "eval", "mode": "fused", "n": 1_000_000, "lobes": 8, "dtype": "bf16",
         "frame": "quat", "norm": "approx", "family": "nasgabor"},
        # Visible primitives only (index list), cosine frames, exact normalisation, an odd number of
        # lobes and of primitives: the paper's "Exact" variant in a renderer that culls first.
        {"name": "visible_cos_l5", "kind": "visible", "n": 400_003, "lobes": 5, "dtype": "f32", "frame": "cos",
         "norm": "exact"},
        # The comparison appearance model: degree-3 spherical harmonics, forward and backward.
        {"name": "sh3_1m", "kind": "sh", "n": 1_000_000, "degree": 3},
        # Scene-scale training: visibility list of one camera, then the fused step on the primitives it sees.
        {"name": "shell_step_6m", "kind": "step", "n": 6_000_000, "lobes": 8, "loss": "given"},
        # Many scenes of uneven size in one persistent launch (16 of them: 4 outputs each).
        {"name": "batched_16", "kind": "batch", "scenes": 16, "n_min": 50_000, "n_max": 3_000_000, "lobes": 0,
         "dtype": "bf16"},
        # Fitting a 16-lobe field to a 4-lobe one at 64 directions: one step.
        {"name": "fit_2m", "kind": "fit", "n": 2_000_000, "lobes": 16, "teacher": 4, "dirs": 64},
        # A small preview image of a small scene: forward only, many short launches.
        {"name": "preview_20k", "kind": "frame", "n": 20_000, "width": 640, "height": 360, "backward": False},
        # Compositing of a full scene at 1080p, forward and backward.
        {"name": "frame_1080p_1m", "kind": "frame", "n": 1_000_000, "width": 1920, "height": 1080, "backward": True},
        # A whole training frame: colours, compositing, image loss, compositing backward, fused step.
        {"name": "train_frame_720p", "kind": "train", "n": 300_000, "lobes": 8, "width": 1280, "height": 720},
        # The fused pass over parameters that live in page-locked host memory.
        {"name": "host_fused_1m", "kind": "host", "n": 1_000_000, "lobes": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("eval", "eval", "eval", "visible", "sh", "step", "batch", "fit", "frame", "frame", "train",
                       "host"))
    if kind == "eval":
        mode = rng.choice(("forward", "autograd", "fused"))
        family = rng.choice(("nasgabor", "nasgabor", "nasg", "sg", "phase")) if mode != "autograd" else "nasgabor"
        return {"kind": kind, "mode": mode, "n": _log_int(rng, 1000, 1_000_000),
                "lobes": rng.choice((1, 2, 3, 4, 5, 6, 8, 8, 12, 16)), "dtype": rng.choice(("f32", "bf16")),
                "frame": rng.choice(("quat", "quat", "cos")) if family == "nasgabor" else "quat",
                "norm": rng.choice(("approx", "approx", "exact")), "family": family}
    if kind == "visible":
        return {"kind": kind, "n": _log_int(rng, 5000, 1_000_000), "lobes": rng.choice((2, 3, 4, 5, 8)),
                "dtype": rng.choice(("f32", "bf16")), "frame": rng.choice(("quat", "cos")),
                "norm": rng.choice(("approx", "exact"))}
    if kind == "sh":
        return {"kind": kind, "n": _log_int(rng, 1000, 2_000_000), "degree": rng.randint(0, 3)}
    if kind == "step":
        return {"kind": kind, "n": _log_int(rng, 20_000, 3_000_000), "lobes": rng.choice((3, 4, 8, 16)),
                "loss": rng.choice(("given", "mse"))}
    if kind == "batch":
        return {"kind": kind, "scenes": rng.randint(2, 16), "n_min": 20_000, "n_max": _log_int(rng, 100_000, 2_000_000),
                "lobes": rng.choice((0, 0, 4, 8)), "dtype": rng.choice(("bf16", "bf16", "f32"))}
    if kind == "fit":
        lobes, teacher = rng.choice(((4, 2), (4, 4), (8, 4), (8, 8), (16, 4)))
        return {"kind": kind, "n": _log_int(rng, 10_000, 1_000_000), "lobes": lobes, "teacher": teacher,
                "dirs": rng.randint(7, 64)}
    if kind == "frame":
        return {"kind": kind, "n": _log_int(rng, 5000, 1_000_000), "width": rng.randint(200, 1920),
                "height": rng.randint(120, 1080), "backward": rng.random() < 0.7}
    if kind == "train":
        return {"kind": kind, "n": _log_int(rng, 10_000, 500_000), "lobes": rng.choice((4, 8)),
                "width": rng.randint(320, 1280), "height": rng.randint(180, 720)}
    return {"kind": kind, "n": _log_int(rng, 20_000, 1_000_000), "lobes": rng.choice((4, 8))}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV)


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV)


def _lobes(g, count, frame="quat", family="nasgabor"):
    """Raw planes [P][count] f32."""
    if frame == "quat":
        q = _randn(g, 4, count)
        rows = [q / q.norm(dim=0, keepdim=True)]
    else:
        ang = 0.02 + _rand(g, 3, count) * (math.pi - 0.04)
        rows = [torch.atanh(torch.cos(ang))]
    shape = {"lam": _rand(g, 1, count) * math.log(1e3),
             "a": torch.log(_rand(g, 1, count).clamp_min(1e-6)),
             "k": torch.atanh((_rand(g, 1, count) * 8.0).clamp_min(1e-6) / 20.0 - 1.0),
             "phi": _rand(g, 1, count) * (2.0 * math.pi)}
    rows += [shape[f] for f in FIELDS[family]]
    rows.append(torch.atanh(_rand(g, 3, count).clamp_max(1.0 - 2.0 ** -20)))
    return torch.cat(rows).contiguous()


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _cloud(case, g):
    """Point cloud in the unit cube seen from (0, 0, 3)."""
    n, lobes = case["n"], case["lobes"]
    return {"params": _lobes(g, n * lobes, case.get("frame", "quat"), case.get("family", "nasgabor")).to(_dtype(case)),
            "c0": _rand(g, 3, n).to(_dtype(case)), "means": _rand(g, n, 3), "g_rgb": _randn(g, n, 3)}


def _morton(p, bits=10):
    lo = p.amin(0)
    q = ((p - lo) / (p.amax(0) - lo).clamp_min(1e-30) * (1 << bits)).long().clamp_max((1 << bits) - 1)
    code = torch.zeros(p.shape[0], dtype=torch.int64, device=DEV)
    for b in range(bits):
        for axis in range(3):
            code |= ((q[:, axis] >> b) & 1) << (3 * b + axis)
    return torch.argsort(code, stable=True)


def _shell(n, g):
    """Noisy sphere shell of radius 1-2 in Morton order."""
    d = _randn(g, n, 3)
    p = d / d.norm(dim=1, keepdim=True) * (1.0 + _rand(g, n, 1))
    return p[_morton(p)].contiguous()


def _ring_camera(seed, means, visible=0.45):
    """A camera on the ring of radius 4, its field of view set so that it sees `visible` of the centres."""
    ang = 2.0 * math.pi * (seed % 8) / 8
    c = (4.0 * math.cos(ang), 4.0 * math.sin(ang), 0.0)
    f = (-math.cos(ang), -math.sin(ang), 0.0)
    r = (-math.sin(ang), math.cos(ang), 0.0)
    r = tuple(-x for x in r)                      # forward x up
    rot = [list(r), [0.0, 0.0, 1.0], list(f)]
    pick = means[:: max(1, means.shape[0] // 200_000)]
    pc = (pick - torch.tensor(c, device=DEV)) @ torch.tensor(rot, device=DEV).T
    t = (pc[:, :2].abs().amax(1) / pc[:, 2].clamp_min(1e-6)).quantile(visible)
    return {"rot": rot, "centre": c, "tan": float(t)}


def _train_state(g, n, lobes):
    """A training state in mid-training."""
    count = n * lobes
    master, c0 = _lobes(g, count), _rand(g, 3, n)
    return nb.TrainState(master, c0, m=_randn(g, 10, count).mul_(1e-3), v=_rand(g, 10, count).mul_(1e-4),
                         c0_m=_randn(g, 3, n).mul_(1e-3), c0_v=_rand(g, 3, n).mul_(1e-4))


def _batch_sizes(case, seed):
    """The scenes' sizes, log-uniform; they are the case's own, the same for every seed."""
    g = torch.Generator()
    g.manual_seed(1000 * case["scenes"] + case["n_max"] % 997)
    u = torch.rand(case["scenes"], generator=g).tolist()
    pick = torch.randint(0, 3, (case["scenes"],), generator=g).tolist()
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
    return [(int(math.exp(lo + x * (hi - lo))), case["lobes"] or (4, 8, 16)[j]) for x, j in zip(u, pick)]


def _frame_geometry(g, n):
    spacing = 3.0 / n ** (1.0 / 3.0)              # of the centres in their cube
    return {"means": _rand(g, n, 3) * 3.0 - 1.5,
            "scales": torch.exp(_rand(g, n, 3) * 2.0 - 2.0) * spacing,
            "quats": _randn(g, n, 4), "opacity": _rand(g, n) * 0.9 + 0.05}


def _frame_camera(case):
    fx = 0.5 * case["width"] / FRAME_TAN
    return nb.raster_camera([[1, 0, 0], [0, 1, 0], [0, 0, 1]], CENTRE_FRAME, case["width"], case["height"], fx)


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = {"case": case}
    if kind == "eval":
        s.update(_cloud(case, g))
        if case["mode"] == "autograd":
            for k in ("params", "c0", "means"):
                s[k].requires_grad_(True)
        return s
    if kind == "visible":
        s.update(_cloud(case, g))
        s["means"] = _shell(case["n"], g)
        cam = _ring_camera(seed, s["means"])
        idx, count = nb.nasg_frustum_compact(s["means"], cam["rot"], cam["centre"], cam["tan"])
        n = case["n"]
        s.update(cam=cam["centre"], idx=idx[: int(count)].contiguous(), rgb=torch.zeros((n, 3), device=DEV),
                 g_params=torch.zeros(s["params"].shape, device=DEV), g_c0=torch.zeros((3, n), device=DEV),
                 g_means=torch.zeros((n, 3), device=DEV))
        return s
    if kind == "sh":
        n = case["n"]
        s.update(coeffs=_randn(g, (case["degree"] + 1) ** 2, 3, n) * 0.3, means=_rand(g, n, 3), g_rgb=_randn(g, n, 3))
        return s
    if kind == "step":
        n = case["n"]
        s["means"] = _shell(n, g)
        s["cam"] = _ring_camera(seed, s["means"])
        s["upstream"] = _randn(g, n, 3) if case["loss"] == "given" else _rand(g, n, 3)
        s["state"] = _train_state(g, n, case["lobes"])
        s["rgb"] = torch.zeros((n, 3), device=DEV)
        s["idx"] = torch.zeros(n, device=DEV, dtype=torch.int32)
        s["count"] = torch.zeros(1, device=DEV, dtype=torch.int32)
        s["workspace"] = torch.empty(nb.nasg_frustum_workspace_bytes(n), device=DEV, dtype=torch.uint8)
        s["t"] = FIRST_STEP
        return s
    if kind == "batch":
        scenes = []
        for n, lobes in _batch_sizes(case, seed):
            sc = _cloud({"n": n, "lobes": lobes, "dtype": case["dtype"]}, g)
            sc.update(cam=CENTRE_CLOUD, n_lobes=lobes)
            scenes.append(sc)
        s["scenes"] = scenes
        s["batch"] = nb.Batch(scenes)
        s["batch"].autotune(reps=3)
        return s
    if kind == "fit":
        n = case["n"]
        s["state"] = _train_state(g, n, case["lobes"])
        s["teacher"] = _lobes(g, n * case["teacher"])
        s["teacher_c0"] = _rand(g, 3, n)
        d = _randn(g, case["dirs"], 3)
        s["dirs"] = (d / d.norm(dim=1, keepdim=True)).contiguous()
        s["loss"] = torch.zeros(1, device=DEV)
        s["workspace"] = torch.empty(int(nb.lib.nasgabor_fit_workspace_bytes()), device=DEV, dtype=torch.uint8)
        s["t"] = FIRST_STEP
        return s
    if kind in ("frame", "train"):
        n = case["n"]
        s.update(_frame_geometry(g, n))
        s["raster"] = nb.Raster(n, _frame_camera(case), PAIR_CAP if n >= 100_000 else PAIR_CAP >> 3)
        shape = (case["height"], case["width"], 3)
        if kind == "frame":
            s["colours"] = _rand(g, n, 3)
            s["g_image"] = _randn(g, *shape) * (2.0 / (shape[0] * shape[1] * 3))
        else:
            s["state"] = _train_state(g, n, case["lobes"])
            s["target"] = _rand(g, *shape)
            s["t"] = FIRST_STEP
        return s
    # page-locked host arrays
    c = _cloud({"n": case["n"], "lobes": case["lobes"], "dtype": "bf16"}, g)
    for k, v in c.items():
        s[k] = v.cpu().pin_memory()
    n = case["n"]
    s["out"] = tuple(torch.zeros(shape).pin_memory() for shape in ((n, 3), tuple(c["params"].shape), (3, n), (n, 3)))
    s["fused"] = nb.HostFused(n, case["lobes"])
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def _state_out(st):
    return {"master": st.master, "m": st.m, "v": st.v, "params_bf16": st.params_bf16, "c0": st.c0_master,
            "c0_m": st.c0_m, "c0_v": st.c0_v, "c0_bf16": st.c0_bf16}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "eval":
        lobes = case["lobes"]
        if case["mode"] == "forward":
            return nb.nasgabor_eval_fwd(s["params"], s["c0"], s["means"], CENTRE_CLOUD, lobes, frame_mode=case["frame"],
                                        norm_mode=case["norm"], family=case["family"])
        if case["mode"] == "autograd":
            s["params"].grad = s["c0"].grad = s["means"].grad = None
            rgb = nb.NasgEval.apply(s["params"], s["c0"], s["means"], CENTRE_CLOUD, lobes, case["frame"], case["norm"])
            rgb.backward(s["g_rgb"])
            return rgb, s["params"].grad, s["c0"].grad, s["means"].grad
        return nb.nasgabor_fused_fwd_bwd(s["params"], s["c0"], s["means"], CENTRE_CLOUD, s["g_rgb"], lobes,
                                         frame_mode=case["frame"], norm_mode=case["norm"], family=case["family"])
    if kind == "visible":
        args = dict(frame_mode=case["frame"], norm_mode=case["norm"], idx=s["idx"])
        nb.nasgabor_eval_fwd(s["params"], s["c0"], s["means"], s["cam"], case["lobes"], rgb=s["rgb"], **args)
        nb.nasgabor_eval_bwd(s["params"], s["means"], s["cam"], s["g_rgb"], case["lobes"], g_params=s["g_params"],
                             g_c0=s["g_c0"], g_means=s["g_means"], **args)
        return s["rgb"], s["g_params"], s["g_c0"], s["g_means"]
    if kind == "sh":
        rgb = nb.sh_eval_fwd(s["coeffs"], s["means"], CENTRE_CLOUD, case["degree"])
        g_coeffs, g_means = nb.sh_eval_bwd(s["coeffs"], s["means"], CENTRE_CLOUD, s["g_rgb"], case["degree"])
        return rgb, g_coeffs, g_means
    if kind == "step":
        cam = s["cam"]
        nb.nasg_frustum_compact(s["means"], cam["rot"], cam["centre"], cam["tan"], idx=s["idx"], n_visible=s["count"],
                                workspace=s["workspace"])
        nb.nasgabor_fused_step(s["state"], s["means"], cam["centre"], s["upstream"], case["lobes"], s["t"],
                               idx=s["idx"], n_idx_device=s["count"], rgb=s["rgb"], loss=case["loss"], **ADAM)
        s["t"] += 1
        return {"rgb": s["rgb"], "count": s["count"], **_state_out(s["state"])}
    if kind == "batch":
        s["batch"].run()
        return [[sc["rgb"], sc["g_params"], sc["g_c0"], sc["g_means"]] for sc in s["scenes"]]
    if kind == "fit":
        nb.nasgabor_fit_step(s["state"], s["teacher"], s["teacher_c0"], case["teacher"], s["dirs"], case["lobes"],
                             s["t"], loss=s["loss"], workspace=s["workspace"], **ADAM)
        s["t"] += 1
        return {"loss": s["loss"], **_state_out(s["state"])}
    if kind == "frame":
        r = s["raster"]
        image, final_t = r.forward(s["means"], s["scales"], s["quats"], s["opacity"], s["colours"])
        out = {"image": image, "final_t": final_t, "pairs": r.n_pairs}
        if case["backward"]:
            out["g_colours"], out["g_opacity"] = r.backward(s["colours"], final_t, s["g_image"])
        return out
    if kind == "train":
        r, st, lobes = s["raster"], s["state"], case["lobes"]
        rgb = nb.nasgabor_eval_fwd(st.params_bf16, st.c0_bf16, s["means"], CENTRE_FRAME, lobes)
        image, final_t = r.forward(s["means"], s["scales"], s["quats"], s["opacity"], rgb)
        g_image = (image - s["target"]).mul_(2.0 / s["target"].numel())
        g_colours, g_opacity = r.backward(rgb, final_t, g_image)
        nb.nasgabor_fused_step(st, s["means"], CENTRE_FRAME, g_colours, lobes, s["t"], **ADAM)
        s["t"] += 1
        return {"image": image, "final_t": final_t, "g_colours": g_colours, "g_opacity": g_opacity, **_state_out(st)}
    return s["fused"](s["params"], s["c0"], s["means"], CENTRE_CLOUD, s["g_rgb"], s["out"])


# ---------------------------------------------------------------------------
# The work of one pass
# ---------------------------------------------------------------------------

# FP32 operations of one lobe, counted in its formulas (a transcendental as ten)
FLOPS_FWD, FLOPS_FWD_BWD = 170, 420


def _eval_work(n, n_listed, lobes, planes, es, fwd, bwd):
    b = n_listed * (planes * lobes * es + 12)     # parameters, means
    if fwd:
        b += n_listed * (3 * es + 12)             # c0, colours
    if bwd:
        b += n_listed * (12 + 4 * planes * lobes + 12 + 12)
    return b


def _footprint_pixels(case):
    """About how many (pixel, primitive) contributions a frame has before its pixels stop: the area of the
    alpha >= 1/255 ellipse of a mean primitive at the middle depth, and half of it for what lies behind the stop."""
    n = case["n"]
    fx = 0.5 * case["width"] / FRAME_TAN
    spacing = 3.0 / n ** (1.0 / 3.0)
    mean_s2 = spacing ** 2 * (1.0 - math.exp(-4.0)) / 4.0
    return 0.5 * n * math.pi * 2.0 * math.log(127.0) * (mean_s2 * (fx / 4.0) ** 2 + 0.3)


def _frame_work(case, backward):
    n, pixels = case["n"], case["width"] * case["height"]
    b, f = n * (12 + 12 + 16 + 4 + 12) + pixels * 16, 16 * _footprint_pixels(case)
    if backward:
        b, f = b + n * (12 + 16) + pixels * (12 + 4), f + 45 * _footprint_pixels(case)
    return b, f


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    if kind == "eval":
        planes = (4 if case["frame"] == "quat" else 3) + len(FIELDS[case["family"]]) + 3
        fwd = case["mode"] == "forward"
        es = 2 if case["dtype"] == "bf16" else 4
        b = _eval_work(n, n, case["lobes"], planes, es, True, not fwd)
        if case["mode"] == "autograd":            # the backward runs later, on the inputs it saved
            b += n * (planes * case["lobes"] * es + 12)
        return {"bytes": b, "flops": n * case["lobes"] * (FLOPS_FWD if fwd else FLOPS_FWD_BWD)}
    if kind == "visible":
        planes, es, seen = (10 if case["frame"] == "quat" else 9), 2 if case["dtype"] == "bf16" else 4, 0.45 * n
        return {"bytes": _eval_work(n, seen, case["lobes"], planes, es, True, False)
                + _eval_work(n, seen, case["lobes"], planes, es, False, True) + 8 * seen,
                "flops": seen * case["lobes"] * (FLOPS_FWD + FLOPS_FWD_BWD)}
    if kind == "sh":
        nb_ = (case["degree"] + 1) ** 2
        return {"bytes": n * (nb_ * 12 * 3 + 24 + 36), "flops": n * nb_ * 24}
    if kind == "step":
        seen, scalars = 0.45 * n, 10 * case["lobes"] + 3
        return {"bytes": n * 12 + seen * (8 + 36 + scalars * 26),
                "flops": seen * (case["lobes"] * FLOPS_FWD_BWD + scalars * 14)}
    if kind == "batch":
        es = 2 if case["dtype"] == "bf16" else 4
        sizes = _batch_sizes(case, 0)
        return {"bytes": sum(_eval_work(m, m, lobes, 10, es, True, True) for m, lobes in sizes),
                "flops": sum(m * lobes * FLOPS_FWD_BWD for m, lobes in sizes)}
    if kind == "fit":
        scalars = 10 * case["lobes"] + 3
        return {"bytes": n * (scalars * 26 + (10 * case["teacher"] + 3) * 4),
                "flops": n * (case["dirs"] * (case["lobes"] * FLOPS_FWD_BWD + case["teacher"] * FLOPS_FWD)
                              + scalars * 14)}
    if kind == "frame":
        b, f = _frame_work(case, case["backward"])
        return {"bytes": b, "flops": f}
    if kind == "train":
        b, f = _frame_work(case, True)
        lobes, pixels = case["lobes"], case["width"] * case["height"]
        return {"bytes": b + _eval_work(n, n, lobes, 10, 2, True, False) + pixels * 36
                + n * (24 + (10 * lobes + 3) * 26),
                "flops": f + n * lobes * (FLOPS_FWD + FLOPS_FWD_BWD)}
    return {"bytes": _eval_work(n, n, case["lobes"], 10, 2, True, True), "flops": n * case["lobes"] * FLOPS_FWD_BWD}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------

def _frames64(p, frame):
    if frame == "quat":
        w, x, y, z = p[0:4] / p[0:4].norm(dim=0, keepdim=True)
        return (torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + w * z), 2 * (x * z - w * y)]),
                torch.stack([2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y)]))
    (ct, cp, cs), (st, sp, ss) = torch.tanh(p[0:3]), 1 / torch.cosh(p[0:3])
    return (torch.stack([ct * cp * cs - st * ss, st * cp * cs + ct * ss, -sp * cs]),
            torch.stack([ct * sp, st * sp, cp]))


def _norm64(lam, a, k, phi, norm):
    base = lam * torch.sqrt(1 + a) / math.pi / -torch.expm1(-2 * lam)
    if norm == "approx":
        return base / 2
    big = lam * (1 + a)
    sigma = (big - k) * (big + k)
    pos = sigma > 0
    one = torch.ones_like(sigma)
    r = torch.sqrt(torch.where(pos, sigma, one))
    t = torch.sqrt(torch.where(pos, one, -sigma))
    sinhc = torch.where(pos, (torch.exp(-k * k / (r + big)) - torch.exp(-r - big)) / (2 * r),
                        torch.exp(-big) * torch.sin(t) / t)
    return base / (1 + torch.cos(phi) * (2 * big * sinhc / -torch.expm1(-2 * big)))


def _activate64(p, frame, family):
    """Axes x, z [3][N][L], weights [3][N][L] and (lam, a, k, phi) of raw planes [P][N][L]."""
    x, z = _frames64(p, frame)
    f = 4 if frame == "quat" else 3
    zero = torch.zeros_like(p[0])
    get = {name: p[f + j] for j, name in enumerate(FIELDS[family])}
    lam = torch.exp(get["lam"])
    a = torch.exp(get["a"]) if "a" in get else zero
    k = 20 * (torch.tanh(get["k"]) + 1) if "k" in get else zero
    return x, z, torch.tanh(p[-3:]), lam, a, k, get.get("phi", zero)


def _colour64(p, c0, d, frame, norm, family, extra=0):
    """c0 + sum_l w_l G_l(d); p [P][N][L], c0 [3][N], d [3][N] (or [3][1][D] against [3][N][D] with extra=1)."""
    x, z, w, lam, a, k, phi = _activate64(p, frame, family)
    c = _norm64(lam, a, k, phi, norm)
    if extra:
        x, z, w = x.unsqueeze(-1), z.unsqueeze(-1), w.unsqueeze(-1)
        lam, a, k, phi, c = (t.unsqueeze(-1) for t in (lam, a, k, phi, c))
        d = d[:, None, None, :]
    else:
        d = d.unsqueeze(-1)
    u = (d * z).sum(0)
    v = (d * x).sum(0)
    ln_kappa = torch.log((1 + u) / 2)
    tau = a * v * v / (1 - u * u)
    g = c * torch.exp(2 * lam * torch.expm1((1 + tau) * ln_kappa) + tau * ln_kappa) * (1 + torch.cos(k * v + phi)) / 2
    return torch.stack([c0[j].unsqueeze(-1) + (w[j] * g).sum(1) if extra else c0[j] + (w[j] * g).sum(1)
                        for j in range(3)])


def _chunks(n, lobes, per=3_000_000):
    m = max(1, per // lobes)
    return [slice(i, min(n, i + m)) for i in range(0, n, m)]


def _take(planes, lobes, at):
    return planes.view(planes.shape[0], -1, lobes)[:, at].double()


def _eval64(params, c0, means, cam, g_rgb, lobes, frame="quat", norm="approx", family="nasgabor", rows=None, grads=True):
    """(rgb, g_params, g_c0, g_means), for the listed rows only where given (the others 0)."""
    n = means.shape[0]
    params, c0, means = params.detach(), c0.detach(), means.detach()
    rgb = torch.zeros((n, 3), device=DEV, dtype=torch.float64)
    gp = torch.zeros(params.shape, device=DEV, dtype=torch.float64) if grads else None
    gc = torch.zeros((3, n), device=DEV, dtype=torch.float64)
    gm = torch.zeros((n, 3), device=DEV, dtype=torch.float64)
    cam = torch.tensor(cam, dtype=torch.float32, device=DEV).double()
    total = n if rows is None else rows.shape[0]
    for ch in _chunks(total, lobes):
        at = ch if rows is None else rows[ch]
        p, c, mu = _take(params, lobes, at), c0[:, at].double(), means[at].double()
        for t in (p, c, mu):
            t.requires_grad_(grads)
        r = mu - cam
        d = (r / r.norm(dim=1, keepdim=True)).T
        out = _colour64(p, c, d, frame, norm, family).T
        rgb[at] = out.detach()
        if grads:
            g = torch.autograd.grad(out, (p, c, mu), g_rgb[at].double())
            gp.view(gp.shape[0], n, lobes)[:, at] = g[0]
            gc[:, at], gm[at] = g[1], g[2]
    return rgb, gp, gc, gm


def _sh64(d, degree):
    """Real orthonormal spherical harmonics with the Condon-Shortley phase from their definition."""
    x, y, z = d
    out = []
    # P_l^m(cos t) / sin^m t, and sin^m t (cos, sin)(m p) = Re, Im of (x + i y)^m
    cm, sm = [torch.ones_like(x)], [torch.zeros_like(x)]
    for _ in range(degree):
        cm, sm = cm + [cm[-1] * x - sm[-1] * y], sm + [cm[-1] * y + sm[-1] * x]
    q = {}
    for m in range(degree + 1):
        q[m, m] = torch.full_like(z, float((-1) ** m * math.prod(range(1, 2 * m, 2))))
        if m + 1 <= degree:
            q[m + 1, m] = (2 * m + 1) * z * q[m, m]
        for l in range(m + 2, degree + 1):
            q[l, m] = ((2 * l - 1) * z * q[l - 1, m] - (l + m - 1) * q[l - 2, m]) / (l - m)
    for l in range(degree + 1):
        for m in range(-l, l + 1):
            j = abs(m)
            k = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - j) / math.factorial(l + j))
            out.append(k * q[l, 0] if m == 0 else math.sqrt(2) * k * q[l, j] * (cm[j] if m > 0 else sm[j]))
    return torch.stack(out)


def _adam64(th, m, v, g, t):
    b1, b2 = ADAM["beta1"], ADAM["beta2"]
    m = b1 * m + (1 - b1) * g
    v = b2 * v + (1 - b2) * g * g
    return th - ADAM["lr"] / (1 - b1 ** t) * m / (torch.sqrt(v / (1 - b2 ** t)) + ADAM["eps"]), m, v


def _adam_state64(st, gp, gc, rows, t):
    """The updated state: rows (all where None) of the master, moments and copies move, the others stay."""
    out = {}
    for names, src, g, lobes in ((("master", "m", "v", "params_bf16"), (st.master, st.m, st.v), gp, st.n_lobes),
                                 (("c0", "c0_m", "c0_v", "c0_bf16"), (st.c0_master, st.c0_m, st.c0_v), gc, 1)):
        new = [x.double() for x in src]
        for p in range(g.shape[0]):               # a plane at a time: the states are large
            view = [x[p].view(-1, lobes) for x in new]
            at = slice(None) if rows is None else rows
            th, m, v = _adam64(*(x[at] for x in view), g[p].view(-1, lobes)[at], t)
            view[0][at], view[1][at], view[2][at] = th, m, v
        out.update(zip(names, new))
        out[names[3]] = new[0].to(torch.bfloat16).double()
    return out


def _visible64(means, cam):
    """Rows inside the frustum; the decision is the library's (whole numbers), taken from it."""
    idx, count = nb.nasg_frustum_compact(means, cam["rot"], cam["centre"], cam["tan"])
    return idx[: int(count)].long()


def _project64(s, case):
    mu = s["means"].double() - torch.tensor(CENTRE_FRAME, device=DEV, dtype=torch.float64)
    cam = _frame_camera(case)
    px, py, pz = mu.T
    iz = 1 / pz
    fx, fy = cam.fx, cam.fy
    u, v = cam.cx + fx * px * iz, cam.cy - fy * py * iz
    zero = torch.zeros_like(iz)
    jac = torch.stack([torch.stack([fx * iz, zero, -fx * px * iz * iz], -1),
                       torch.stack([zero, -fy * iz, fy * py * iz * iz], -1)], -2)
    q = s["quats"].double()
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).T
    rot = torch.stack([torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)], -1),
                       torch.stack([2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)], -1),
                       torch.stack([2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1)], -2)
    m = jac @ rot
    cov = (m * s["scales"].double()[:, None, :] ** 2) @ m.transpose(1, 2) + 0.3 * torch.eye(2, device=DEV, dtype=torch.float64)
    return pz, u, v, cov, pz > cam.near_z


def _composite64(s, case, colours, g_of_image):
    """Image, final transmittance and, with g_of_image, the gradients wrt colours and opacities."""
    w, h, tile = case["width"], case["height"], 16
    pz, u, v, cov, valid = _project64(s, case)
    sig = s["opacity"].double()
    a, b, c = cov[:, 0, 0], cov[:, 0, 1], cov[:, 1, 1]
    det = a * c - b * b
    reach = 2 * torch.log((255 * sig).clamp_min(1.0)) * 1.001
    rx, ry = torch.sqrt(a * reach) + 1, torch.sqrt(c * reach) + 1
    tx, ty = (w + tile - 1) // tile, (h + tile - 1) // tile
    lo = lambda t, m: torch.floor(t / tile).clamp(0, m).long()  # noqa: E731
    x0, x1 = lo(u - rx, tx - 1), lo(u + rx, tx - 1)
    y0, y1 = lo(v - ry, ty - 1), lo(v + ry, ty - 1)
    valid = valid & (255 * sig > 1) & (u + rx > 0) & (u - rx < w) & (v + ry > 0) & (v - ry < h)
    order = torch.argsort(s["means"][:, 2] - CENTRE_FRAME[2], stable=True)   # by the f32 depth, ties by index
    order = order[valid[order]]
    nx, ny = (x1 - x0 + 1)[order], (y1 - y0 + 1)[order]
    cnt = nx * ny
    prim = torch.repeat_interleave(order, cnt)
    k = torch.arange(prim.shape[0], device=DEV) - torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt)
    nxr = torch.repeat_interleave(nx, cnt)
    tiles = (y0[prim] + k // nxr) * tx + x0[prim] + k % nxr
    by_tile = torch.argsort(tiles, stable=True)
    prim, tiles = prim[by_tile], tiles[by_tile]
    lens = torch.bincount(tiles, minlength=tx * ty)
    starts = lens.cumsum(0) - lens
    image = torch.zeros((ty * tile, tx * tile, 3), device=DEV, dtype=torch.float64)
    trans = torch.ones((ty * tile, tx * tile), device=DEV, dtype=torch.float64)
    g_c, g_o = torch.zeros_like(colours), torch.zeros_like(sig)
    long_first = torch.argsort(lens, descending=True)
    long_first = long_first[lens[long_first] > 0]
    lens_host = lens[long_first].tolist()
    inside = torch.arange(tile, device=DEV, dtype=torch.float64) + 0.5

    def batches():
        at = 0
        while at < len(lens_host):
            m = max(1, 30_000_000 // (lens_host[at] * tile * tile))
            yield long_first[at:at + m], lens_host[at]
            at += m

    def terms(ids, most):
        j = torch.arange(most, device=DEV)
        real = j[None] < lens[ids][:, None]
        p = prim[(starts[ids][:, None] + j[None]).clamp_max(prim.shape[0] - 1)]              # [tiles, K]
        gx = (ids % tx * tile)[:, None, None] + inside[None, None, :]                        # [tiles, 1, 16]
        gy = (torch.div(ids, tx, rounding_mode="floor") * tile)[:, None, None] + inside[None, :, None]
        px = gx.expand(-1, tile, -1).reshape(len(ids), 1, -1)
        py = gy.expand(-1, -1, tile).reshape(len(ids), 1, -1)
        dx, dy = px - u[p][..., None], py - v[p][..., None]
        q = (c[p][..., None] * dx * dx - 2 * b[p][..., None] * dx * dy + a[p][..., None] * dy * dy) / det[p][..., None]
        rho = torch.exp(-0.5 * q)
        free = sig[p][..., None] * rho
        alpha = free.clamp_max(0.99)
        alpha = torch.where(real[..., None] & (alpha >= 1 / 255), alpha, torch.zeros_like(alpha))
        after = torch.cumprod(1 - alpha, 1)
        alpha = torch.where(after >= 1e-4, alpha, torch.zeros_like(alpha))
        after = torch.cumprod(1 - alpha, 1)
        before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
        return p, rho, free, alpha, before, after

    def pixels(ids):
        r = (torch.div(ids, tx, rounding_mode="floor") * tile)[:, None, None] + torch.arange(tile, device=DEV)[None, :, None]
        q = (ids % tx * tile)[:, None, None] + torch.arange(tile, device=DEV)[None, None, :]
        return r, q

    for ids, most in batches():
        p, _, _, alpha, before, after = terms(ids, most)
        r, q = pixels(ids)
        image[r, q] = torch.einsum("tkp,tkc->tpc", alpha * before, colours[p]).view(len(ids), tile, tile, 3)
        trans[r, q] = after[:, -1].view(len(ids), tile, tile)
    image, trans = image[:h, :w].contiguous(), trans[:h, :w].contiguous()
    if g_of_image is None:
        return image, trans, None, None
    g = torch.zeros((ty * tile, tx * tile, 3), device=DEV, dtype=torch.float64)
    g[:h, :w] = g_of_image(image)
    for ids, most in batches():
        p, rho, free, alpha, before, _ = terms(ids, most)
        r, q = pixels(ids)
        gp = g[r, q].reshape(len(ids), -1, 3)                                                # [tiles, 256, 3]
        wgt = alpha * before
        g_c.index_add_(0, p.reshape(-1), torch.einsum("tkp,tpc->tkc", wgt, gp).reshape(-1, 3))
        dot = torch.einsum("tkc,tpc->tkp", colours[p], gp)
        own = dot * wgt
        later = own.sum(1, keepdim=True) - own.cumsum(1)
        da = dot * before - later / (1 - alpha)
        da = torch.where((alpha > 0) & (free < 0.99), da * rho, torch.zeros_like(da))
        g_o.index_add_(0, p.reshape(-1), da.sum(2).reshape(-1))
    return image, trans, g_c, g_o


def exact(case, seed):
    s = prepare(case, seed)
    kind, lobes = case["kind"], case.get("lobes", 0)
    if kind == "eval":
        grads = case["mode"] != "forward"
        r = _eval64(s["params"], s["c0"], s["means"], CENTRE_CLOUD, s["g_rgb"], lobes, case["frame"], case["norm"],
                    case["family"], grads=grads)
        return r if grads else r[0]
    if kind == "host":
        dev = {k: s[k].to(DEV) for k in ("params", "c0", "means", "g_rgb")}
        r = _eval64(dev["params"], dev["c0"], dev["means"], CENTRE_CLOUD, dev["g_rgb"], lobes)
        return tuple(x.cpu() for x in r)
    if kind == "visible":
        return _eval64(s["params"], s["c0"], s["means"], s["cam"], s["g_rgb"], lobes, case["frame"], case["norm"],
                       rows=s["idx"].long())
    if kind == "sh":
        mu = s["means"].double().requires_grad_(True)
        co = s["coeffs"].double().requires_grad_(True)
        r = mu - torch.tensor(CENTRE_CLOUD, device=DEV, dtype=torch.float64)
        rgb = torch.einsum("jcn,jn->nc", co, _sh64((r / r.norm(dim=1, keepdim=True)).T, case["degree"]))
        g = torch.autograd.grad(rgb, (co, mu), s["g_rgb"].double(), allow_unused=True)
        return rgb.detach(), g[0], torch.zeros_like(mu) if g[1] is None else g[1]
    if kind == "batch":
        return [list(_eval64(sc["params"], sc["c0"], sc["means"], CENTRE_CLOUD, sc["g_rgb"], sc["n_lobes"]))
                for sc in s["scenes"]]
    if kind == "step":
        st, cam = s["state"], s["cam"]
        rows = _visible64(s["means"], cam)
        values = (st.params_bf16, st.c0_bf16, s["means"], cam["centre"])
        up = s["upstream"]
        if case["loss"] == "mse":
            rgb = _eval64(*values, None, lobes, rows=rows, grads=False)[0]
            up = 2 * (rgb - up.double()) / (3 * rows.shape[0])
        rgb, gp, gc, _ = _eval64(*values, up, lobes, rows=rows)
        return {"rgb": rgb, "count": None, **_adam_state64(st, gp, gc, rows, s["t"])}
    if kind == "fit":
        return _fit64(s, case)
    if kind == "frame":
        g = (lambda image: s["g_image"].double()) if case["backward"] else None
        image, trans, g_c, g_o = _composite64(s, case, s["colours"].double(), g)
        out = {"image": image, "final_t": trans, "pairs": None}
        if case["backward"]:
            out.update(g_colours=g_c, g_opacity=g_o)
        return out
    st = s["state"]
    values = (st.params_bf16, st.c0_bf16, s["means"], CENTRE_FRAME)
    rgb = _eval64(*values, None, lobes, grads=False)[0]
    target = s["target"].double()
    image, trans, g_c, g_o = _composite64(s, case, rgb, lambda im: (im - target) * (2.0 / target.numel()))
    _, gp, gc, _ = _eval64(*values, g_c, lobes)
    return {"image": image, "final_t": trans, "g_colours": g_c, "g_opacity": g_o,
            **_adam_state64(st, gp, gc, None, s["t"])}


def _fit64(s, case):
    st, n, lobes, teacher = s["state"], case["n"], case["lobes"], case["teacher"]
    d = s["dirs"].double().T
    d = (d / d.norm(dim=0, keepdim=True)).contiguous()   # unit but for their storage in 32 bits
    gp = torch.zeros(st.master.shape, device=DEV, dtype=torch.float64)
    gc = torch.zeros((3, n), device=DEV, dtype=torch.float64)
    loss = torch.zeros((), device=DEV, dtype=torch.float64)
    for at in _chunks(n, lobes * case["dirs"], 20_000_000):
        with torch.no_grad():
            want = _colour64(_take(s["teacher"], teacher, at), s["teacher_c0"][:, at].double(), d, "quat", "approx",
                             "nasgabor", extra=1)
        p, c = _take(st.params_bf16, lobes, at).requires_grad_(True), st.c0_bf16[:, at].double().requires_grad_(True)
        err = (_colour64(p, c, d, "quat", "approx", "nasgabor", extra=1) - want).square().sum() / (3 * case["dirs"])
        g = torch.autograd.grad(err, (p, c))
        gp.view(10, n, lobes)[:, at], gc[:, at] = g[0], g[1]
        loss += err.detach() / n
    return {"loss": loss.reshape(1), **_adam_state64(st, gp, gc, None, s["t"])}
