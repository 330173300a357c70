"""Performance cases: the calls a program that renders or trains Gaussian
splats makes through ``paper_2604_02120_gb300.gs``, from the smallest frame to
a 3840x2160 training step.

A case is a dict of plain values.  Its ``kind`` is the entry point:

* ``render_small``    gs_render_small: a small scene's frame in one launch
* ``render``          gs.render: project -> bin/sort -> blend of one frame
* ``step``            BatchRenderer's captured graph: forward + backward of all views
* ``project``         gs.project / gs_project_views
* ``project_backward`` gs.project_backward
* ``bin_sort``        BinSorter.run (full rectangles, keys, synchronising) or
                      gs_bin_sort_views (opacity-aware, no synchronisation)
* ``blend_forward``, ``blend_backward``  the blend of given lists and its gradient
* ``blend_autograd``  BlendFunction under torch.autograd (forward + backward)

The scenes are the repository's own recipes (``scenes.py``: uniform,
clustered, heavy-tailed), drawn on the GPU so that a case is made quickly.  The
blend and bin/sort cases get their splats from a projection written here in
64 bits (rounded to float32), so that ``exact`` can work from the same inputs
without the package.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_02120_gb300 import gs, scenes

DEV = "cuda"
# the scene recipes of scenes.py
RECIPES = ("uniform", "clustered", "heavy")


# ------------------------------------------------------------------- the list

def _case(kind, recipe, n, width, height, **kw):
    c = dict(kind=kind, recipe=recipe, n=n, width=width, height=height, sh_degree=0, views=1, variant="fp16_split",
             tight=False, longest_first=False, bg=0.0, max_per_tile=1024, capacity=0)
    c.update(kw)
    return c


def listed():
    return [
        # a preview or thumbnail frame of a small asset: latency is all that counts
        dict(_case("render_small", "uniform", 10_000, 256, 256), name="render_small_256x256_10k"),
        # one interactive viewer frame, the README's call
        dict(_case("render", "uniform", 200_000, 1280, 720, sh_degree=3, capacity=3_000_000),
             name="render_1280x720_200k"),
        # a training step at the benchmark's workload: one 4K view, 3M heavy-tailed Gaussians
        dict(_case("step", "heavy", 3_000_000, 3840, 2160, sh_degree=3, variant="bf16_split", tight=True,
                   longest_first=True, capacity=170_000_000), name="step_3840x2160_3m"),
        # a training step over a batch of cameras of uneven resolution (the ring of 16 views)
        dict(_case("step", "clustered", 1_500_000, 0, 0, views=16, longest_first=True, capacity=260_000_000),
             name="step_16_views_1500k"),
        # preprocessing alone, with view-dependent colour
        dict(_case("project", "heavy", 3_000_000, 3840, 2160, sh_degree=3), name="project_3m_sh3"),
        # its gradient, the last stage of a training step
        dict(_case("project_backward", "clustered", 1_000_000, 1920, 1080, sh_degree=3),
             name="project_backward_1m_sh3"),
        # binning of the 4K step, opacity-aware lists, as a captured step calls it
        dict(_case("bin_sort", "heavy", 3_000_000, 3840, 2160, tight=True, capacity=170_000_000),
             name="bin_sort_tight_3840x2160_3m"),
        # binning of one 1080p frame: full rectangles with sorted keys, synchronising
        dict(_case("bin_sort", "clustered", 1_000_000, 1920, 1080, capacity=20_000_000),
             name="bin_sort_full_1920x1080_1m"),
        # the blend of a dense 1080p frame
        dict(_case("blend_forward", "clustered", 1_000_000, 1920, 1080, variant="bf16_split", longest_first=True),
             name="blend_forward_1920x1080_1m"),
        # its gradient
        dict(_case("blend_backward", "clustered", 1_000_000, 1920, 1080, variant="bf16_split", longest_first=True),
             name="blend_backward_1920x1080_1m"),
        # the differentiable blend as a PyTorch training loop uses it
        dict(_case("blend_autograd", "uniform", 200_000, 1280, 720, bg=0.5), name="blend_autograd_1280x720_200k"),
        # the same with the float32 CUDA-core variant, the default of gs_blend_opts
        dict(_case("blend_autograd", "uniform", 50_000, 641, 479, variant="fp32"), name="blend_fp32_641x479_50k"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render_small", "render", "step", "project", "project_backward", "bin_sort", "bin_sort",
                       "blend_forward", "blend_backward", "blend_autograd"])
    deg = rng.choice([0, 1, 2, 3])
    if kind == "render_small":
        n, w, h = _log_int(rng, 500, 16_000), _log_int(rng, 48, 400), _log_int(rng, 48, 400)
        per_tile = 24 * n * 1.6 / (((w + 15) // 16) * ((h + 15) // 16))
        cap = 256
        while cap < min(n, per_tile + 64):
            cap *= 2
        return _case(kind, "uniform", n, w, h, sh_degree=deg, max_per_tile=cap)
    recipe = rng.choice(RECIPES)
    w, h = _log_int(rng, 100, 3840), _log_int(rng, 100, 2160)
    n = _log_int(rng, 2_000, 3_000_000 if kind in ("project", "project_backward", "bin_sort", "step") else 1_000_000)
    kw = dict(sh_degree=deg if kind in ("render", "step", "project", "project_backward") else 0)
    if kind in ("render", "step", "blend_forward", "blend_backward", "blend_autograd"):
        kw["variant"] = rng.choice(["fp16_split", "fp16_split", "bf16_split", "bf16_split", "fp32", "fp16", "bf16"])
        kw["bg"] = rng.choice([0.0, 0.5])
    if kind in ("step", "bin_sort", "blend_forward", "blend_backward"):
        # the heavy-tailed scenes' full rectangles would cost more than any listed case
        kw["tight"] = True if recipe == "heavy" else rng.random() < 0.5
        kw["longest_first"] = kind != "bin_sort" and rng.random() < 0.7
    if recipe == "heavy" and not kw.get("tight", False):
        n = min(n, 50_000)
    if kind in ("step", "project", "project_backward"):
        v = rng.choice([1, 1, 2, 5])
        kw["views"] = v
        n = max(2_000, min(n, 2_000_000 // v if v > 1 else n))
    c = _case(kind, recipe, n, w, h, **kw)
    # the instances a program provides for: three times the recipe's mean (clusters near the camera)
    c["capacity"] = 100_000 + int(3 * sum(_sample_instances(c, cam) for cam in _cameras(c, 0)) * n)
    return c


# ------------------------------------------------------------------ the inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + 17)
    return g


def _scene(case, seed):
    """The recipe's 3D Gaussians as float32 tensors on the GPU."""
    g, n, recipe = _gen(seed), case["n"], case["recipe"]
    kw = dict(device=DEV, dtype=torch.float32, generator=g)
    k = (case["sh_degree"] + 1) ** 2
    if recipe == "uniform":
        means = torch.rand(n, 3, **kw) * 2 - 1
        ls = torch.randn(n, 3, **kw) * 0.5 - 4.0
    else:
        centres = torch.rand(64, 3, **kw) * 4 - 2
        member = torch.randint(0, 64, (n,), device=DEV, generator=g)
        means = centres[member] + torch.randn(n, 3, **kw) * 0.2
        if recipe == "clustered":
            ls = torch.randn(n, 3, **kw) * 0.8 - 4.5
            axis = torch.randint(0, 3, (n, 1), device=DEV, generator=g)
            ls.scatter_add_(1, axis, torch.full((n, 1), -2.0, device=DEV))
        else:  # Student-t with 3 degrees of freedom; capped where float32 covariances would overflow
            chi = torch.randn(n, 3, **kw) ** 2 + torch.randn(n, 3, **kw) ** 2 + torch.randn(n, 3, **kw) ** 2
            ls = (-4.5 + 0.7 * torch.randn(n, 3, **kw) / (chi / 3).clamp_min(1e-12).sqrt()).clamp(-20.0, 10.0)
    quats = torch.nn.functional.normalize(torch.randn(n, 4, **kw), dim=1)
    if recipe == "heavy":  # Beta(0.5, 0.5): the arcsine law
        opac = (torch.sin(torch.rand(n, **kw) * (math.pi / 2)) ** 2).clamp(1e-7, 1 - 1e-7)
    else:
        opac = torch.sigmoid(torch.randn(n, **kw))
    sh = torch.randn(n, k, 3, **kw) * 0.05
    sh[:, 0, :] *= 6.0  # DC ~ N(0, 0.3)
    return dict(means=means.contiguous(), scales=ls.exp().contiguous(), quats=quats.contiguous(),
                opacities=opac.contiguous(), sh=sh.contiguous(), sh_degree=case["sh_degree"])


def _cameras(case, seed):
    if case["views"] == 1:
        return [scenes.look_at_camera((0, 0, -3), (0, 0, 0), case["width"], case["height"])]
    rng = np.random.default_rng(int(seed))
    if case["width"] == 0:  # the ring of mixed resolutions
        choices = [(640, 480), (1280, 720), (1600, 900), (1920, 1080)]
        # every resolution equally often, in a seeded order: the work does not depend on the seed
        res = [choices[i % 4] for i in rng.permutation(case["views"])]
    else:
        w, h = case["width"], case["height"]
        res = [(max(16, w >> (i % 2)), max(16, h >> (i % 2))) for i in range(case["views"])]
    return scenes.ring_cameras(case["views"], 3.0, res)


def _sh_basis(d, deg):
    """Real spherical harmonics of unit directions, columns in (l, m) order."""
    x, y, z = d.unbind(1)
    b = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if deg >= 1:
        c = math.sqrt(3 / (4 * math.pi))
        b += [-c * y, c * z, -c * x]
    if deg >= 2:
        c = 0.5 * math.sqrt(15 / math.pi)
        b += [c * x * y, -c * y * z, 0.25 * math.sqrt(5 / math.pi) * (2 * z * z - x * x - y * y), -c * x * z,
              0.5 * c * (x * x - y * y)]
    if deg >= 3:
        c33, c32 = 0.25 * math.sqrt(35 / (2 * math.pi)), 0.5 * math.sqrt(105 / math.pi)
        c31, c30 = 0.25 * math.sqrt(21 / (2 * math.pi)), 0.25 * math.sqrt(7 / math.pi)
        b += [-c33 * y * (3 * x * x - y * y), c32 * x * y * z, -c31 * y * (4 * z * z - x * x - y * y),
              c30 * z * (2 * z * z - 3 * x * x - 3 * y * y), -c31 * x * (4 * z * z - x * x - y * y),
              0.5 * c32 * z * (x * x - y * y), -c33 * x * (x * x - 3 * y * y)]
    return torch.stack(b, 1)


def _project64(means, scales, quats, sh, deg, cam):
    """EWA projection in 64 bits: mean2d, conic, depth, radius, rgb, live (differentiable)."""
    R = torch.tensor(np.float32(cam.R), device=means.device).double()
    t = torch.tensor(np.float32(cam.t), device=means.device).double()
    fx, fy, cx, cy = (float(np.float32(v)) for v in (cam.fx, cam.fy, cam.cx, cam.cy))
    low = float(np.float32(cam.lowpass))
    p = means @ R.T + t
    x, y, z = p.unbind(1)
    live = z > float(np.float32(cam.znear))
    z = torch.where(live, z, torch.ones_like(z))
    qw, qx, qy, qz = torch.nn.functional.normalize(quats, dim=1).unbind(1)
    rot = torch.stack([1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - qw * qz), 2 * (qx * qz + qw * qy),
                       2 * (qx * qy + qw * qz), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - qw * qx),
                       2 * (qx * qz - qw * qy), 2 * (qy * qz + qw * qx), 1 - 2 * (qx * qx + qy * qy)], 1)
    M = rot.view(-1, 3, 3) * scales[:, None, :]
    zero = torch.zeros_like(z)
    J = torch.stack([fx / z, zero, -fx * x / (z * z), zero, fy / z, -fy * y / (z * z)], 1).view(-1, 2, 3)
    U = (J @ R) @ M
    a = (U[:, 0] * U[:, 0]).sum(1) + low
    b = (U[:, 0] * U[:, 1]).sum(1)
    c = (U[:, 1] * U[:, 1]).sum(1) + low
    det = a * c - b * b
    live = live & (det > 0)
    det = torch.where(live, det, torch.ones_like(det))
    conic = torch.stack([c / det, -b / det, a / det], 1)
    mean2d = torch.stack([fx * x / z + cx, fy * y / z + cy], 1)
    with torch.no_grad():
        live = live & (mean2d.abs() <= 2.0 ** 23).all(1)
        lam = 0.5 * (a + c) + (0.25 * (a - c) ** 2 + b * b).sqrt()
        r = torch.where(live, (3 * lam.sqrt()).ceil().clamp(max=2.0 ** 24), zero).long()
        x0, x1, y0, y1 = _rect(mean2d, r, cam.width, cam.height)
        live = live & (x0 <= x1) & (y0 <= y1)
        radius = torch.where(live, r, torch.zeros_like(r)).int()
    d = torch.nn.functional.normalize(means - (-(R.T @ t)), dim=1)
    rgb = ((sh * _sh_basis(d, deg)[:, :, None]).sum(1) + 0.5).clamp_min(0)
    return mean2d, conic, p[:, 2], radius, rgb, live


def _rect(mean2d, r, w, h):
    m = mean2d.floor().long()
    q = [torch.div(v, 16, rounding_mode="floor") for v in (m[:, 0] - r, m[:, 0] + r, m[:, 1] - r, m[:, 1] + r)]
    return (q[0].clamp(min=0), q[1].clamp(max=(w + 15) // 16 - 1), q[2].clamp(min=0),
            q[3].clamp(max=(h + 15) // 16 - 1))


def _masked(x, live):
    return torch.where(live.view(-1, *([1] * (x.dim() - 1))), x, torch.zeros_like(x))


def _exact_projection(sc, cam):
    with torch.no_grad():
        m, c, d, r, rgb, live = _project64(sc["means"].double(), sc["scales"].double(), sc["quats"].double(),
                                           sc["sh"].double(), sc["sh_degree"], cam)
        return dict(mean2d=_masked(m, live), conic=_masked(c, live), depth=d, radius=r, rgb=_masked(rgb, live))


def _splats(case, seed, cam):
    """The splats of a projection (float32) that the blend and bin/sort cases take."""
    sc = _scene(case, seed)
    s = _exact_projection(sc, cam)
    out = {k: (v if k == "radius" else v.float()).contiguous() for k, v in s.items()}
    out["opacity"] = sc["opacities"]
    return out


def _upstream(shape, seed):
    return torch.randn(shape, device=DEV, generator=_gen(seed + 7919))


def _opts(case, order=None):
    return gs.make_opts(case["variant"], bg=(case["bg"],) * 3, tile_order=order)


def _sorter(case):
    """A sorter whose buffers already fit the scene, as a program's do after its first frames; the
    buffers' unused ends are zero, so that they can be returned whole."""
    srt = gs.BinSorter(DEV, capacity=case["capacity"])
    srt.keys.zero_()
    srt.ids.zero_()
    return srt


def _instance_count(n_views, n, mean2d, radius, depth, widths, heights, conic, pmin):
    """The instances a sort of these items has (a call that finds its capacity too small reports them)."""
    cap = 1 << 16
    ws = torch.empty(gs.gs_bin_sort_workspace_size(n_views * n, cap, widths[0], heights[0]) + 256, device=DEV,
                     dtype=torch.uint8)
    ids = torch.empty(cap, device=DEV, dtype=torch.int32)
    ranges = torch.empty(2 * sum(gs.num_tiles(w, h) for w, h in zip(widths, heights)), device=DEV, dtype=torch.int32)
    _, count = gs.gs_bin_sort_views(n_views, n, mean2d, radius, depth, widths, heights, cap, ws, None, ids, ranges,
                                    check=False, conic=conic, power_min=pmin)
    return count


def _lists(case, s, cam):
    """Tile lists of one view's splats, as the program has them before it blends."""
    if not case["tight"]:
        return gs.BinSorter(DEV, capacity=1 << 20).run(s["mean2d"], s["radius"], s["depth"], cam.width, cam.height)
    pmin = gs.alpha_power_min(s["opacity"])
    args = (1, case["n"], s["mean2d"], s["radius"], s["depth"], [cam.width], [cam.height])
    cap = max(1, _instance_count(*args, s["conic"], pmin))
    ws = torch.empty(gs.gs_bin_sort_workspace_size(case["n"], cap, cam.width, cam.height) + 256, device=DEV,
                     dtype=torch.uint8)
    ids = torch.zeros(cap, device=DEV, dtype=torch.int32)
    ranges = torch.empty(2 * gs.num_tiles(cam.width, cam.height), device=DEV, dtype=torch.int32)
    gs.gs_bin_sort_views(*args, cap, ws, None, ids, ranges, conic=s["conic"], power_min=pmin)
    return dict(ids=ids, tile_ranges=ranges)


def prepare(case, seed):
    kind = case["kind"]
    cams = _cameras(case, seed)
    cam, n = cams[0], case["n"]
    f32, i32 = dict(device=DEV, dtype=torch.float32), dict(device=DEV, dtype=torch.int32)
    st = dict(case=case, cams=cams)
    if kind == "render_small":
        st["scene"] = _scene(case, seed)
        W, H, nt = cam.width, cam.height, gs.num_tiles(cam.width, cam.height)
        st["cam"] = gs.make_camera(cam)
        st["out"] = dict(mean2d=torch.empty(n, 2, **f32), conic=torch.empty(n, 3, **f32), depth=torch.empty(n, **f32),
                         radius=torch.empty(n, **i32), rgb=torch.empty(n, 3, **f32), touched=torch.empty(n, **i32),
                         ids=torch.zeros(nt * case["max_per_tile"], **i32), ranges=torch.empty(2 * nt, **i32),
                         image=torch.empty(3, H, W, **f32), T_final=torch.empty(H, W, **f32),
                         n_contrib=torch.empty(H, W, **i32))
    elif kind == "render":
        st["scene"] = _scene(case, seed)
        st["opts"] = _opts(case)
        st["sorter"] = _sorter(case)
    elif kind == "step":
        sc = st["scene"] = _scene(case, seed)
        r = gs.BatchRenderer(sc, cams, _opts(case), case["capacity"], DEV, longest_first=case["longest_first"],
                             opacity_aware=case["tight"])
        r.ids.zero_()
        r.dL.copy_(_upstream((3 * r.pixels,), seed))
        r.capture()
        st["renderer"] = r
    elif kind == "project":
        st["scene"] = _scene(case, seed)
        if len(cams) > 1:
            V = len(cams)
            st["gs_cams"] = [gs.make_camera(c) for c in cams]
            st["out"] = dict(mean2d=torch.empty(V * n, 2, **f32), conic=torch.empty(V * n, 3, **f32),
                             depth=torch.empty(V * n, **f32), radius=torch.empty(V * n, **i32),
                             rgb=torch.empty(V * n, 3, **f32), touched=torch.empty(V * n, **i32))
    elif kind == "project_backward":
        sc = st["scene"] = _scene(case, seed)
        st["gs_cams"] = [gs.make_camera(c) for c in cams]
        st["radius"] = torch.cat([_exact_projection(sc, c)["radius"] for c in cams]).contiguous()
        V = len(cams)
        st["g"] = dict(zip(("mean2d", "conic", "rgb"), _projection_grads(V * n, seed)))
    elif kind == "bin_sort":
        s = st["splats"] = _splats(case, seed, cam)
        if case["tight"]:
            st["pmin"] = gs.alpha_power_min(s["opacity"])
            cap = case["capacity"]
            need = gs.gs_bin_sort_workspace_size(n, cap, cam.width, cam.height)
            st["workspace"] = torch.empty(need + 256, device=DEV, dtype=torch.uint8)
            st["ids"] = torch.zeros(cap, **i32)
            st["ranges"] = torch.empty(2 * gs.num_tiles(cam.width, cam.height), **i32)
            st["count"] = torch.zeros(1, device=DEV, dtype=torch.int64)
        else:
            st["sorter"] = _sorter(case)
    else:
        s = st["splats"] = _splats(case, seed, cam)
        st["bs"] = _lists(case, s, cam)
        order = None
        if case["longest_first"]:
            order = st["order"] = gs.tile_order(st["bs"]["tile_ranges"], [cam.width], [cam.height])
        st["opts"] = _opts(case, order)
        if kind != "blend_forward":
            st["dL"] = _upstream((3, cam.height, cam.width), seed)
        if kind == "blend_backward":
            st["fwd"] = gs.blend_forward(cam.width, cam.height, st["bs"], s, s["opacity"], st["opts"])
        if kind == "blend_autograd":
            st["leaves"] = [s[k].clone().requires_grad_(True) for k in ("mean2d", "conic", "opacity", "rgb")]
    return st


def _projection_grads(items, seed):
    g = _gen(seed + 31)
    # the sizes a blend's gradients have against each other: pixels, conic entries, colours
    return [torch.randn(items, k, device=DEV, generator=g) * s for k, s in ((2, 0.1), (3, 1.0), (3, 1.0))]


# --------------------------------------------------------------------- the pass

def run(state):
    case, kind, cams = state["case"], state["case"]["kind"], state["cams"]
    cam, n = cams[0], case["n"]
    if kind == "render_small":
        sc, o = state["scene"], state["out"]
        gs.gs_render_small(n, sc["means"], sc["scales"], sc["quats"], sc["sh"], sc["sh_degree"], state["cam"], None,
                           case["max_per_tile"], sc["opacities"], (case["bg"],) * 3, o["mean2d"], o["conic"],
                           o["depth"], o["radius"], o["rgb"], o["touched"], o["ids"], o["ranges"], o["image"],
                           o["T_final"], o["n_contrib"])
        return o
    if kind == "render":
        r = gs.render(state["scene"], cam, state["opts"], state["sorter"])
        p, b, f = r["project"], r["bin_sort"], r["blend"]
        return dict(image=f["image"], T_final=f["T_final"], n_contrib=f["n_contrib"], mean2d=p["mean2d"],
                    conic=p["conic"], depth=p["depth"], radius=p["radius"], rgb=p["rgb"],
                    touched=p["tiles_touched"], keys=state["sorter"].keys, ids=state["sorter"].ids,
                    ranges=b["tile_ranges"], count=b["n_instances"])
    if kind == "step":
        r = state["renderer"]
        r.graph.replay()
        return dict(image=r.image, T_final=r.T, n_contrib=r.nc, dmean2d=r.g_mean2d, dconic=r.g_conic,
                    dopacity=r.g_opac, drgb=r.g_rgb, ids=r.ids, ranges=r.ranges, count=r.count)
    if kind == "project":
        sc = state["scene"]
        if len(cams) == 1:
            p = gs.project(sc["means"], sc["scales"], sc["quats"], sc["sh"], sc["sh_degree"], cam)
            return dict(mean2d=p["mean2d"], conic=p["conic"], depth=p["depth"], radius=p["radius"], rgb=p["rgb"],
                        touched=p["tiles_touched"])
        o = state["out"]
        gs.gs_project_views(n, sc["means"], sc["scales"], sc["quats"], sc["sh"], sc["sh_degree"], state["gs_cams"],
                            o["mean2d"], o["conic"], o["depth"], o["radius"], o["rgb"], o["touched"])
        return o
    if kind == "project_backward":
        sc, g = state["scene"], state["g"]
        return gs.project_backward(sc["means"], sc["scales"], sc["quats"], sc["sh"], sc["sh_degree"],
                                   state["gs_cams"], state["radius"], g["mean2d"], g["conic"], g["rgb"])
    s = state["splats"]
    if kind == "bin_sort":
        if case["tight"]:
            gs.gs_bin_sort_views(1, n, s["mean2d"], s["radius"], s["depth"], [cam.width], [cam.height],
                                 case["capacity"], state["workspace"], None, state["ids"], state["ranges"],
                                 count_dev=state["count"], conic=s["conic"], power_min=state["pmin"])
            return dict(ids=state["ids"], ranges=state["ranges"], count=state["count"])
        b = state["sorter"].run(s["mean2d"], s["radius"], s["depth"], cam.width, cam.height)
        return dict(keys=state["sorter"].keys, ids=state["sorter"].ids, ranges=b["tile_ranges"],
                    count=b["n_instances"])
    if kind == "blend_forward":
        return gs.blend_forward(cam.width, cam.height, state["bs"], s, s["opacity"], state["opts"])
    if kind == "blend_backward":
        return gs.blend_backward(cam.width, cam.height, state["bs"], s, s["opacity"], state["opts"], state["fwd"],
                                 state["dL"])
    leaves, bs = state["leaves"], state["bs"]
    image, T, nc = gs.BlendFunction.apply(*leaves, bs["tile_ranges"], gs._list_ids(bs), cam.width, cam.height,
                                          state["opts"])
    dm, dc, do, drgb = torch.autograd.grad(image, leaves, state["dL"])
    return dict(image=image.detach(), T_final=T, n_contrib=nc, dmean2d=dm, dconic=dc, dopacity=do, drgb=drgb)


# ------------------------------------------------------------------ the floors

# Evaluated pairs per pixel of the recipes' dense frames (sum of n_contrib over
# the pixels, measured once per recipe at the listed sizes): early termination
# and the scene's coverage hold it there however many splats there are.
_PAIRS_PER_PIXEL = {("uniform", False): 106.0, ("uniform", True): 60.0, ("clustered", False): 440.0,
                    ("clustered", True): 130.0, ("heavy", False): 650.0, ("heavy", True): 45.0}


def _sample_instances(case, cam):
    """Instances per Gaussian, from 2048 of the recipe's Gaussians projected in numpy."""
    rng = np.random.default_rng(0)
    m = 2048
    if case["recipe"] == "uniform":
        means, ls = rng.uniform(-1, 1, (m, 3)), rng.normal(-4.0, 0.5, (m, 3))
    else:
        means = rng.uniform(-2, 2, (64, 3))[rng.integers(0, 64, m)] + rng.normal(0, 0.2, (m, 3))
        if case["recipe"] == "clustered":
            ls = rng.normal(-4.5, 0.8, (m, 3))
            ls[np.arange(m), rng.integers(0, 3, m)] -= 2.0
        else:
            ls = np.clip(-4.5 + 0.7 * rng.standard_t(3.0, (m, 3)), -20, 10)
    p = means @ np.asarray(cam.R).T + np.asarray(cam.t)
    z = np.where(p[:, 2] > cam.znear, p[:, 2], np.inf)
    sig = np.exp(ls) * (cam.fy / z)[:, None]  # pixels, along each axis seen face on
    r = 3 * np.sqrt((sig ** 2).max(1) + cam.lowpass)
    u, v = cam.fx * p[:, 0] / z + cam.cx, cam.fy * p[:, 1] / z + cam.cy

    def span(c, ext, size):
        lo, hi = np.floor((c - ext) / 16), np.floor((c + ext) / 16)
        return np.maximum(0, np.minimum(hi, (size + 15) // 16 - 1) - np.maximum(lo, 0) + 1)

    full = np.where(np.isfinite(z), span(u, r, cam.width) * span(v, r, cam.height), 0)
    if not case["tight"]:
        return float(full.mean())
    # opacity-aware: about the area of the splat's visible ellipse in tiles, plus its outline's
    mid = np.sort(sig, 1)
    area = math.pi * 3.0 * np.sqrt((mid[:, 2] ** 2 + 0.3) * (mid[:, 1] ** 2 + 0.3)) * 2.0
    est = float(np.minimum(full, area / 256 + 2.0 * r / 16 + 1).mean())
    # most of a needle splat's ellipse lies outside the image (measured: 0.25 to 0.28 of the estimate)
    return 0.27 * est if case["recipe"] == "heavy" else est


def work(case):
    kind, n, k = case["kind"], case["n"], (case["sh_degree"] + 1) ** 2
    cams = _cameras(case, 0)
    pix = sum(c.width * c.height for c in cams)
    tiles = sum(c.num_tiles for c in cams)
    items = n * len(cams)
    inst = sum(_sample_instances(case, c) * n for c in cams)
    pairs = min(256.0 * inst, _PAIRS_PER_PIXEL[case["recipe"], case["tight"]] * pix)
    scene = n * (40 + 12 * k)
    splat, proj_flops = 44, n * len(cams) * (150.0 + 6.0 * k)
    # a blend reads each splat once, at most the ids whose pairs it evaluates, and writes 20 bytes per pixel
    used = min(inst, pairs / 64.0)
    fwd = dict(bytes=36 * n * len(cams) + 4 * used + 20 * pix, flops=22.0 * pairs)
    bwd = dict(bytes=72 * n * len(cams) + 4 * used + 20 * pix, flops=60.0 * pairs)
    sort_bytes = 12 * items + (16 * items if case["tight"] else 0) + 4 * inst + 8 * tiles
    if kind == "project":
        b, f = scene - 4 * n + splat * items, proj_flops
    elif kind == "project_backward":
        b, f = 2 * (scene - 4 * n) + 36 * items, 3 * proj_flops
    elif kind == "bin_sort":
        b, f = sort_bytes + (0 if case["tight"] else 8 * inst), 0.0
    elif kind == "blend_forward":
        b, f = fwd["bytes"], fwd["flops"]
    elif kind == "blend_backward":
        b, f = bwd["bytes"], bwd["flops"]
    elif kind == "blend_autograd":
        b, f = fwd["bytes"] + bwd["bytes"], fwd["flops"] + bwd["flops"]
    elif kind == "step":
        b = scene + 32 * items + 4 * inst + 20 * pix + 12 * pix
        f = proj_flops + fwd["flops"] + bwd["flops"]
    else:  # a frame
        b, f = scene + splat * items + (12 if kind == "render" else 4) * inst + 8 * tiles + 20 * pix, \
            proj_flops + fwd["flops"]
    return {"bytes": int(b), "flops": int(f)}


# ------------------------------------------------------------- the exact result

def _box_max(A, B, C, bx0, bx1, by0, by1):
    """Largest -q/2 over the box of offsets, q = A dx^2 + 2 B dx dy + C dy^2 (A, C > 0)."""
    q = torch.full_like(A, math.inf)
    for ex in (bx0, bx1):
        dy = torch.minimum(torch.maximum(-B * ex / C, by0), by1)
        q = torch.minimum(q, A * ex * ex + 2 * B * ex * dy + C * dy * dy)
    for ey in (by0, by1):
        dx = torch.minimum(torch.maximum(-B * ey / A, bx0), bx1)
        q = torch.minimum(q, A * dx * dx + 2 * B * dx * ey + C * ey * ey)
    inside = (bx0 <= 0) & (bx1 >= 0) & (by0 <= 0) & (by1 >= 0)
    return torch.where(inside, torch.zeros_like(q), -0.5 * q)


def _exact_lists(s, w, h, cull):
    """Tile lists in (tile, depth, index) order: sorted ids, start and count per
    tile.  cull drops pairs whose alpha stays below 1/255 over the whole tile
    (they change nothing)."""
    tx = (w + 15) // 16
    nt = tx * ((h + 15) // 16)
    m = s["mean2d"].double()
    r = s["radius"].long()
    order = torch.sort(s["depth"].float(), stable=True).indices
    order = order[r[order] > 0]
    x0, x1, y0, y1 = (v[order] for v in _rect(m, r, w, h))
    wid = (x1 - x0 + 1).clamp(min=0)
    cnt = wid * (y1 - y0 + 1).clamp(min=0)
    cum = torch.cumsum(cnt, 0)
    con, o = s["conic"].double(), s["opacity"].double()
    pmin = torch.log(1.0 / (255.0 * o)) - 1e-6
    tiles, ids = [], []
    total = int(cum[-1]) if cum.numel() else 0
    b0, nb = 0, cnt.numel()
    while b0 < nb and total:
        done = int(cum[b0 - 1]) if b0 else 0
        b1 = max(b0 + 1, int(torch.searchsorted(cum, done + (1 << 24), right=True)))
        c = cnt[b0:b1]
        rep = torch.repeat_interleave(torch.arange(b0, b1, device=m.device), c)
        off = torch.arange(rep.numel(), device=m.device) - (cum[rep] - cnt[rep] - done)
        ty = y0[rep] + torch.div(off, wid[rep], rounding_mode="floor")
        txx = x0[rep] + off % wid[rep]
        g = order[rep]
        if cull:
            A, B, C = con[g].unbind(1)
            bx, by = m[g, 0] - 16.0 * txx, m[g, 1] - 16.0 * ty
            keep = (_box_max(A, B, C, bx - 15.5, bx - 0.5, by - 15.5, by - 0.5) >= pmin[g]) & (o[g] >= 1 / 256)
            keep |= ~((A > 0) & (C > 0))
            ty, txx, g = ty[keep], txx[keep], g[keep]
        tiles.append((ty * tx + txx).int())
        ids.append(g.int())
        b0 = b1
    if not tiles:
        z = torch.zeros(0, device=m.device, dtype=torch.int64)
        return z, torch.zeros(nt, device=m.device, dtype=torch.int64), torch.zeros(nt, device=m.device,
                                                                                   dtype=torch.int64)
    tile, idx = torch.sort(torch.cat(tiles), stable=True)
    ids = torch.cat(ids)[idx]
    count = torch.bincount(tile.long(), minlength=nt)
    return ids, torch.cumsum(count, 0) - count, count


def _exact_blend(s, w, h, bg, dL=None, chunk=64, group=1024):
    """Image, T_final (and, with dL, the gradients) of the blend in 64 bits."""
    ids, start, count = _exact_lists(s, w, h, True)
    dev, tx = start.device, (w + 15) // 16
    n = s["opacity"].numel()
    mean, con, o, rgb = (s[k].double() for k in ("mean2d", "conic", "opacity", "rgb"))
    image = torch.zeros(3, h, w, device=dev, dtype=torch.float64)
    Tim = torch.ones(h, w, device=dev, dtype=torch.float64)
    gr = None
    if dL is not None:
        gr = [torch.zeros(n, k, device=dev, dtype=torch.float64) for k in (2, 3, 1, 3)]
    torder = torch.sort(count, descending=True).indices
    lp = torch.arange(256, device=dev)

    def walk(tiles, px, py, g, total):
        """One front-to-back walk; with g (upstream, B x 256 x 3) and total, also the gradients."""
        B = tiles.numel()
        T = torch.ones(B, 256, device=dev, dtype=torch.float64)
        col = torch.zeros(B, 256, 3, device=dev, dtype=torch.float64)
        done = torch.zeros(B, 256, device=dev, dtype=torch.bool)
        pre = torch.zeros(B, 256, device=dev, dtype=torch.float64)
        act, pos = torch.arange(B, device=dev), 0
        while True:
            act = act[(count[tiles[act]] > pos) & ~done[act].all(1)]
            if act.numel() == 0:
                return T, col
            t = tiles[act]
            j = pos + torch.arange(chunk, device=dev)
            ok = j[None, :] < count[t][:, None]
            gi = ids[(start[t][:, None] + j[None, :]).clamp(max=ids.numel() - 1)].long()
            A, Bc, C = (con[gi][:, :, i, None] for i in range(3))
            dx = mean[gi][:, :, 0, None] - px[act][:, None, :]
            dy = mean[gi][:, :, 1, None] - py[act][:, None, :]
            pw = -0.5 * (A * dx * dx + C * dy * dy) - Bc * dx * dy
            e = torch.exp(pw.clamp(max=0))
            raw = o[gi][:, :, None] * e
            al = raw.clamp(max=0.99)
            use = (al >= 1 / 255) & ok[:, :, None] & ~done[act][:, None, :]
            a = torch.where(use, al, torch.zeros_like(al))
            Ti = T[act][:, None, :] * torch.cumprod(1 - a, 1)
            alive = Ti >= 1e-4
            Tp = torch.cat([T[act][:, None, :], Ti[:, :-1]], 1)
            a = torch.where(alive, a, torch.zeros_like(a))
            wt = a * Tp
            col[act] += torch.einsum("blp,blc->bpc", wt, rgb[gi])
            if g is not None:
                cg = torch.einsum("blc,bpc->blp", rgb[gi], g[act])
                wc = wt * cg
                incl = pre[act][:, None, :] + torch.cumsum(wc, 1)
                pre[act] = incl[:, -1]
                live = a > 0
                dal = torch.where(live, Tp * cg - (total[act][:, None, :] - incl) / (1 - a), torch.zeros_like(a))
                un = live & (raw <= 0.99)
                dal = torch.where(un, dal, torch.zeros_like(dal))
                dp = torch.where(pw <= 0, dal * al, torch.zeros_like(dal))
                flat = gi.reshape(-1)
                red = [torch.stack([-(dp * (A * dx + Bc * dy)).sum(2), -(dp * (Bc * dx + C * dy)).sum(2)], 2),
                       torch.stack([-0.5 * (dp * dx * dx).sum(2), -(dp * dx * dy).sum(2),
                                    -0.5 * (dp * dy * dy).sum(2)], 2),
                       (dal * e).sum(2)[:, :, None], torch.einsum("blp,bpc->blc", wt, g[act])]
                for acc, v in zip(gr, red):
                    acc.index_add_(0, flat, torch.where(ok[:, :, None], v, torch.zeros_like(v)).reshape(-1, v.shape[2]))
            T[act] = torch.where(alive, Ti, torch.full_like(Ti, math.inf)).amin(1).minimum(T[act])
            done[act] |= ~alive[:, -1]
            pos += chunk

    for b in range(0, torder.numel(), group):
        tiles = torder[b:b + group]
        ix = (tiles % tx)[:, None] * 16 + (lp & 15)[None, :]
        iy = torch.div(tiles, tx, rounding_mode="floor")[:, None] * 16 + (lp >> 4)[None, :]
        inside = (ix < w) & (iy < h)
        px, py = ix.double() + 0.5, iy.double() + 0.5
        T, col = walk(tiles, px, py, None, None)
        full = col + T[:, :, None] * bg
        yy, xx = iy[inside], ix[inside]
        image[:, yy, xx] = full[inside].T
        Tim[yy, xx] = T[inside]
        if dL is not None:
            g = torch.zeros_like(col)
            g[inside] = dL.double()[:, yy, xx].T
            walk(tiles, px, py, g, (full * g).sum(2))
    if gr is not None:
        gr[2] = gr[2][:, 0]
    return image, Tim, gr


def _with_opacity(p, sc):
    return dict(p, opacity=sc["opacities"])


def exact(case, seed):
    with torch.no_grad():
        kind, cams = case["kind"], _cameras(case, seed)
        cam = cams[0]
        bg = case["bg"]
        if kind == "bin_sort":
            return None  # whole numbers only
        if case["variant"] in ("fp16", "bf16"):
            return None  # single-term operands: the exponent is rounded on purpose
        if case["recipe"] == "heavy" and kind in ("render", "step"):
            return None  # needle splats: a float32 conic is not near the 64-bit one, nor then the image
        if kind == "project":
            ps = [_exact_projection(_scene(case, seed), c) for c in cams]
            out = {k: torch.cat([p[k] for p in ps]) for k in ("mean2d", "conic", "depth", "rgb")}
            # the needle splats' conics are ill-conditioned: float32 covariances do not determine them
            conic = None if case["recipe"] == "heavy" else out["conic"]
            return dict(mean2d=out["mean2d"], conic=conic, depth=out["depth"], radius=None, rgb=out["rgb"],
                        touched=None)
        if kind == "project_backward":
            return _exact_project_backward(case, seed, cams)
        if kind in ("render", "render_small"):
            sc = _scene(case, seed)
            p = _exact_projection(sc, cam)
            image, T, _ = _exact_blend(_with_opacity(p, sc), cam.width, cam.height, bg)
            f = dict(image=image, T_final=T, n_contrib=None)
            q = dict(mean2d=p["mean2d"], conic=p["conic"], depth=p["depth"], radius=None, rgb=p["rgb"], touched=None)
            if kind == "render":
                return dict(f, **q, keys=None, ids=None, ranges=None, count=None)
            return dict(q, ids=None, ranges=None, **f)
        if kind == "step":
            if len(cams) * case["n"] > 4_000_000:
                return None  # sixteen dense views would take longer than a check may
            sc = _scene(case, seed)
            pix = sum(c.width * c.height for c in cams)
            dL, off = _upstream((3 * pix,), seed), 0
            img, Ts, grads = [], [], []
            for c in cams:
                np_ = c.width * c.height
                d = dL[3 * off:3 * (off + np_)].view(3, c.height, c.width)
                image, T, g = _exact_blend(_with_opacity(_exact_projection(sc, c), sc), c.width, c.height, bg, d)
                img.append(image.reshape(-1))
                Ts.append(T.reshape(-1))
                grads.append(g)
                off += np_
            return dict(image=torch.cat(img), T_final=torch.cat(Ts), n_contrib=None,
                        dmean2d=torch.cat([g[0] for g in grads]),
                        dconic=torch.cat([g[1] for g in grads]) if case["recipe"] == "uniform" else None,
                        dopacity=sum(g[2] for g in grads), drgb=torch.cat([g[3] for g in grads]), ids=None,
                        ranges=None, count=None)
        s = _splats(case, seed, cam)
        dL = None if kind == "blend_forward" else _upstream((3, cam.height, cam.width), seed)
        image, T, g = _exact_blend(s, cam.width, cam.height, bg, dL)
        f = dict(image=image, T_final=T, n_contrib=None)
        if kind == "blend_forward":
            return f
        if case["recipe"] != "uniform":
            # a needle splat's conic gradient sums the squared distance of far pixels, where one
            # pixel at the 1/255 threshold outweighs all the others
            g[1] = None
        if kind == "blend_backward":
            return dict(mean2d=g[0], conic=g[1], opacity=g[2], rgb=g[3])
        return dict(f, dmean2d=g[0], dconic=g[1], dopacity=g[2], drgb=g[3])


def _exact_project_backward(case, seed, cams):
    sc = _scene(case, seed)
    n, V = case["n"], len(cams)
    if case["recipe"] == "heavy":
        return None  # needle splats: the inverse of a float32 covariance has no digits to compare
    gm, gc, gr = (g.double() for g in _projection_grads(V * n, seed))
    leaves = [sc[k].double().requires_grad_(True) for k in ("means", "scales", "quats", "sh")]
    out = [torch.zeros_like(v) for v in leaves]
    for v, cam in enumerate(cams):
        with torch.enable_grad():
            m, c, _, _, rgb, live = _project64(*leaves, case["sh_degree"], cam)
            sl = slice(v * n, (v + 1) * n)
            gv = [_masked(x[sl], live) for x in (gm, gc, gr)]
            part = torch.autograd.grad([m, c, rgb], leaves, gv)
        for acc, x in zip(out, part):
            acc += _masked(x, live)
    return dict(dmeans=out[0], dscales=out[1], dquats=out[2], dsh=out[3])
