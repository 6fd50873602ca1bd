"""The work that users of this rasterizer have it do, as cases that can be timed and compared.

Every case is a call (or the few calls) a user's program makes through the package's public entry
points: whole frames with a `Renderer`, training steps with `render_gaussians`, the sorting stage
alone, the differentiable blending stage alone (`rasterize`), a scheduled batch of views
(`MultiView`) and the tile-cost model's forward and backward.  Scenes follow the distributions of
`paper_2505_24796_gb300.scenes` (a uniform box, anisotropic clusters, an opaque-in-faint volume), drawn
on the GPU from the seed alone.

`exact` evaluates the same definitions in 64 bits with plain torch: projection, coverage by the
projected square, front-to-back blending per pixel, and their derivatives by autograd.
"""
import math

import numpy as np
import torch

import paper_2505_24796_gb300 as tc
from paper_2505_24796_gb300 import scenes, sched

DEV = "cuda"
SQRT_PI = math.sqrt(math.pi)


def listed():
    return [
        # A thumbnail or a probe view: the whole frame is launch latency (the plain workload).
        dict(name="frame_128", kind="frame", scene="box", width=128, height=128, P=1000, sh=0, fx=128.0),
        # An interactive viewer's frame of a trained-looking scene (the headline workload).
        dict(name="frame_1080p", kind="frame", scene="cluster", width=1920, height=1080, P=1_000_000, sh=3, fx=1100.0),
        # A ragged size (neither side a multiple of the tile), a faint and narrow scene, the opacity-aware
        # squares: a viewer window that the user has dragged to some size.
        dict(name="frame_1237x701", kind="frame", scene="cluster", width=1237, height=701, P=301_317, sh=2, fx=900.0,
             tight=True),
        # An offline 4K frame of a large scene with wide footprints: 600M splats.
        dict(name="frame_4k", kind="frame", scene="box_cluster", width=3840, height=2160, P=6_000_000, sh=3, fx=2200.0),
        # One optimisation step at 720p (the differentiation workload): forward, loss, backward to the
        # 3D parameters.
        dict(name="train_720p", kind="train", scene="box", width=1280, height=720, P=500_000, sh=0, fx=1280.0),
        # One optimisation step on a full-HD photograph with degree-3 colours, as 3DGS training runs.
        dict(name="train_1080p", kind="train", scene="cluster", width=1920, height=1080, P=1_000_000, sh=3, fx=1100.0),
        # The first steps of a training on a small ragged image: launches and host calls count.
        dict(name="train_200x136", kind="train", scene="box", width=200, height=136, P=3000, sh=1, fx=200.0),
        # The sorting stage with the 3-sigma squares (tcgs_bin_sort), for a program with its own renderer.
        dict(name="sort_1600x900", kind="sort", scene="cluster", width=1600, height=900, P=800_000, sh=0, fx=900.0),
        # The blending stage alone, forward and backward, at its default precision (FP32), between a
        # program's own projection and loss.
        dict(name="blend_fp32_1024x512", kind="blend", scene="cluster", width=1024, height=512, P=250_000, sh=0, fx=587.0,
             precision="fp32"),
        # Sixteen low-resolution views of one scene in one scheduled launch (reinforcement learning,
        # previews): features, predicted costs, queue order and the batched render.
        dict(name="views_16x320x240", kind="views", views=16, width=320, height=240, faint=200_000, blobs=60),
        # One gradient evaluation of the tile-cost model on the tiles of 16 full-size views.
        dict(name="cost_model_56k", kind="model", rows=56_048),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "train", "train", "sort", "blend", "views", "model"])
    if kind == "model":
        return dict(kind="model", rows=_log_uniform(rng, 300, 56_048))
    if kind == "views":
        return dict(kind="views", views=rng.randint(2, 16), width=rng.randint(96, 320), height=rng.randint(80, 240),
                    faint=_log_uniform(rng, 20_000, 200_000), blobs=rng.randint(5, 60))
    width = _log_uniform(rng, 100, 1920)
    height = max(65, min(1080, int(width * rng.uniform(0.5, 0.75))))
    scene = rng.choice(["box", "cluster"])
    most = 250_000 if scene == "box" else 1_000_000
    # as many Gaussians as such a view has in earnest: more for larger images, over a factor of about 60
    P = max(500, min(most, int(width * height * math.exp(rng.uniform(math.log(0.02), math.log(1.2))))))
    case = dict(kind=kind, scene=scene, width=width, height=height, P=P, sh=rng.randint(0, 3),
                fx=round(width * rng.uniform(0.55, 1.0), 1))
    if kind == "frame":
        case["tight"] = rng.random() < 0.3
    if kind == "sort":
        case["exact_tiles"] = rng.random() < 0.5
    if kind == "blend":
        case["precision"] = rng.choice(["fp32", "tc_fp16_split"])
    return case


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) + 7919)


def _rand(g, *shape, lo=0.0, hi=1.0):
    return torch.rand(*shape, generator=g, device=DEV) * (hi - lo) + lo


def _randn(g, *shape, mean=0.0, std=1.0):
    return torch.randn(*shape, generator=g, device=DEV) * std + mean


def _camera(case):
    return scenes.pinhole(case["width"], case["height"], case["fx"])


def _sh(g, P, degree):
    sh = _randn(g, P, (degree + 1) ** 2, 3, std=0.05)
    sh[:, 0] = _rand(g, P, 3, lo=-SQRT_PI, hi=SQRT_PI)   # colour uniform in [0, 1]
    return sh


def _box(g, P, degree):
    """The plain and differentiation workloads' recipe: wide footprints, mid opacities."""
    means = torch.stack([_rand(g, P, lo=-2.0, hi=2.0), _rand(g, P, lo=-2.0, hi=2.0), _rand(g, P, lo=2.0, hi=10.0)], 1)
    return dict(means3=means.contiguous(), scales=torch.exp(_randn(g, P, 3, mean=-3.0, std=0.5)), quats=_randn(g, P, 4),
                opacity=torch.sigmoid(_randn(g, P)), sh=_sh(g, P, degree), sh_degree=degree)


def _clusters(g, P, degree, cam, wide, spread_of_scales):
    """The precision workload's recipe (64 clusters in the frustum, small splats, bimodal opacity), or with
    `wide` the large workload's (256 clusters in a box, large splats, mid opacities)."""
    n = 256 if wide else 64
    if wide:
        centres = torch.stack([_rand(g, n, lo=-2.0, hi=2.0), _rand(g, n, lo=-2.0, hi=2.0), _rand(g, n, lo=2.0, hi=10.0)], 1)
        spread = _rand(g, n, 3, lo=0.02, hi=0.3)
    else:
        z = _rand(g, n, lo=4.0, hi=40.0)
        x = z * _rand(g, n, lo=-0.75, hi=0.75) * (cam["width"] / 2.0) / cam["fx"]
        y = z * _rand(g, n, lo=-0.75, hi=0.75) * (cam["height"] / 2.0) / cam["fy"]
        centres = torch.stack([x, y, z], 1)
        spread = z[:, None] * _rand(g, n, 3, lo=0.01, hi=0.08)
    axes = torch.linalg.qr(_randn(g, n, 3, 3))[0]
    label = torch.randint(0, n, (P,), generator=g, device=DEV)
    local = _randn(g, P, 3) * spread[label]
    means = centres[label] + (axes[label] * local[:, None, :]).sum(2)
    if wide:
        means[:, :2].clamp_(-2.0, 2.0)
        means[:, 2].clamp_(2.0, 10.0)
        opacity = torch.sigmoid(_randn(g, P))
        scales = torch.exp(_randn(g, P, 3, mean=-3.0, std=0.5))
    else:
        means[:, 2].clamp_(1.0, 50.0)
        opaque = _rand(g, P) < 0.7
        opacity = torch.where(opaque, torch.sigmoid(_randn(g, P, mean=3.0)), torch.sigmoid(_randn(g, P, mean=-3.0)))
        scales = torch.exp(_randn(g, P, 3, mean=-4.5, std=spread_of_scales))
    return dict(means3=means.contiguous(), scales=scales, quats=_randn(g, P, 4), opacity=opacity, sh=_sh(g, P, degree),
                sh_degree=degree)


def _scene(case, seed):
    g, cam = _gen(seed), _camera(case)
    if case["scene"] == "box":
        return cam, _box(g, case["P"], case["sh"])
    # scenes in training hold fewer needles (whose gradients cancel to less than 32 bits hold) than finished ones
    return cam, _clusters(g, case["P"], case["sh"], cam, case["scene"] == "box_cluster",
                          0.6 if case["kind"] in ("train", "blend") else 1.0)


def _target(case, seed):
    """A smooth image in [0, 1], as a photograph is at the scale of a splat."""
    small = torch.rand(1, 3, 9, 16, generator=_gen(seed + 1), device=DEV)
    size = (case["height"], case["width"])
    return torch.nn.functional.interpolate(small, size=size, mode="bicubic", align_corners=True)[0].clamp(0, 1).contiguous()


def _capacity(case):
    """Splats that the sorting stage's caller makes room for, with 20 to 50% to spare (its buffers outlive a scene)."""
    per = 3.0 + 6.0 * (case["fx"] / 320.0) ** 1.8 if case["scene"] == "box" else 3.0 + 5.0 * (case["fx"] / 1520.0) ** 1.5
    return int(case["P"] * per) + 20_000


def _occluded(case, seed):
    """The occluded-volume workload: a faint volume with opaque clusters inside it, from a sphere of cameras."""
    g = _gen(seed)
    nf, nb = case["faint"], case["blobs"] * 3000
    centre = torch.tensor(scenes.SCENE_CENTRE, dtype=torch.float32, device=DEV)
    u = _randn(g, nf, 3)
    faint = centre + u / u.norm(dim=1, keepdim=True) * (6.0 * _rand(g, nf) ** (1.0 / 3.0))[:, None]
    c = centre + _rand(g, case["blobs"], 3, lo=-4.2, hi=4.2)
    blob = c[torch.randint(0, case["blobs"], (nb,), generator=g, device=DEV)] + _randn(g, nb, 3)
    P = nf + nb
    scene = dict(means3=torch.cat([faint, blob]).contiguous(), scales=torch.exp(_randn(g, P, 3, mean=-2.3, std=0.3)),
                 quats=_randn(g, P, 4),
                 opacity=torch.cat([torch.sigmoid(_randn(g, nf, mean=-3.0, std=0.5)), torch.sigmoid(_randn(g, nb, mean=4.0))]),
                 sh=_sh(g, P, 0), sh_degree=0)
    return scenes.low_res_cameras(case["views"], int(seed) + 1000, case["width"], case["height"]), scene


def _model_inputs(case, seed):
    """Feature rows as tcgs_tile_features makes them, and log costs that depend on them."""
    g, n = _gen(seed), case["rows"]
    length = torch.log1p(torch.exp(_randn(g, n, mean=5.5, std=1.3)).floor())
    x = torch.stack([length, _rand(g, n, lo=0.05, hi=0.8), _rand(g, n, lo=0.6, hi=1.0), _rand(g, n, lo=0.0, hi=2.2),
                     _randn(g, n, mean=-3.0, std=1.5), length + _randn(g, n, std=0.4),
                     torch.full((n,), math.log(1280.0 * 720.0), device=DEV) + 0.5 * _randn(g, n).sign(),
                     torch.where(_rand(g, n) < 0.95, 1.0, 0.5)], 1).contiguous()
    y = (x[:, 0] - 1.5 * x[:, 1] + 0.1 * _randn(g, n)).clamp_min(0.0).contiguous()
    return x, y


def prepare(case, seed):
    kind = case["kind"]
    if kind == "model":
        x, y = _model_inputs(case, seed)
        return dict(case=case, x=x, y=y, model=sched.TileCostModel(DEV, seed=int(seed) % 1000), norm=tc.tcgs_feature_norm(x),
                    grad=torch.zeros(1377, device=DEV), loss=torch.zeros(1, device=DEV))
    if kind == "views":
        cams, scene = _occluded(case, seed)
        views = sched.MultiView(scene, cams)
        model = sched.TileCostModel(DEV, seed=int(seed) % 1000)
        model.fit(*views.training_data(), steps=20)
        return dict(case=case, views=views, model=model)
    cam, scene = _scene(case, seed)
    if kind == "train":
        target = _target(case, seed)
        leaves = {k: scene[k].requires_grad_(True) for k in ("means3", "scales", "quats", "opacity", "sh")}
        return dict(case=case, cam=cam, leaves=leaves, target=target)
    # what a user knows of a scene before rendering: the projection's tile counts size the splat buffer
    tight = bool(case.get("tight"))
    proj = tc.tcgs_project(cam, scene["means3"], scene["scales"], scene["quats"], scene["sh"], scene["sh_degree"],
                           opacity=scene["opacity"] if tight else None)
    capacity = int(proj["tiles_touched"].to(torch.int64).sum().item())
    if kind == "frame":
        return dict(case=case, scene=scene, r=tc.Renderer(cam, case["P"], capacity + 1024, device=DEV, tight_radius=tight))
    gw, gh = tc.grid(cam)
    if kind == "sort":
        capacity = _capacity(case)
    out = dict(ids_sorted=torch.zeros(max(capacity, 1), dtype=torch.int32, device=DEV),
               tile_ranges=torch.empty(gw * gh, 2, dtype=torch.int32, device=DEV),
               n_splats=torch.empty(1, dtype=torch.int64, device=DEV),
               status=torch.empty(1, dtype=torch.int32, device=DEV))
    if kind == "sort":
        ws = torch.empty(tc.tcgs_bin_sort_workspace_size(case["P"], capacity, gw * gh), dtype=torch.uint8, device=DEV)
        return dict(case=case, cam=tc.make_camera(cam), proj=proj, opacity=scene["opacity"], capacity=capacity, ws=ws, out=out)
    tc.tcgs_bin_sort_exact(cam, proj["mean2d"], proj["radius"], proj["depth"], proj["conic"], scene["opacity"], capacity, out=out)
    leaves = dict(mean2d=proj["mean2d"], conic=proj["conic"], opacity=scene["opacity"], rgb=proj["rgb"])
    leaves = {k: v.requires_grad_(True) for k, v in leaves.items()}
    weight = _randn(_gen(seed + 1), 3, case["height"], case["width"])
    return dict(case=case, cam=cam, leaves=leaves, bins=out, weight=weight)


# ---------------------------------------------------------------- one pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "frame":
        r = state["r"]
        out = r.frame(state["scene"])
        return dict(out, n_splats=r.bins["n_splats"])
    if kind == "train":
        p = state["leaves"]
        for v in p.values():
            v.grad = None
        img, T = tc.render_gaussians(state["cam"], p["means3"], p["scales"], p["quats"], p["opacity"], p["sh"], case["sh"])
        (img - state["target"]).abs().mean().backward()
        return dict(img=img.detach(), T=T.detach(), **{"d" + k: v.grad for k, v in p.items()})
    if kind == "sort":
        p = state["proj"]
        exact = bool(case.get("exact_tiles"))
        return tc.tcgs_bin_sort(state["cam"], p["mean2d"], p["radius"], p["depth"], state["capacity"], workspace=state["ws"],
                                out=state["out"], conic=p["conic"] if exact else None,
                                opacity=state["opacity"] if exact else None)
    if kind == "blend":
        p = state["leaves"]
        for v in p.values():
            v.grad = None
        img, T = tc.rasterize(p["mean2d"], p["conic"], p["opacity"], p["rgb"], state["cam"], state["bins"]["tile_ranges"],
                              state["bins"]["ids_sorted"], precision=case["precision"])
        img.backward(state["weight"])
        return dict(img=img.detach(), T=T.detach(), **{"d" + k: v.grad for k, v in p.items()})
    if kind == "views":
        views = state["views"]
        views.render(views.queue("mlp", state["model"]))
        return [dict(v.out) for v in views.views]
    state["grad"].zero_()
    state["loss"].zero_()
    cost = tc.tcgs_mlp_fwd(state["model"].params, state["norm"], state["x"])
    tc.tcgs_mlp_bwd(state["model"].params, state["norm"], state["x"], state["y"], grad=state["grad"], loss=state["loss"])
    return dict(cost=cost, grad=state["grad"], loss=state["loss"])


# ---------------------------------------------------------------- the work of a pass

def work(case):
    """Bytes: inputs and outputs once each.  Operations: the projection's and the blending's, the latter for
    about as many pixel-Gaussian pairs as such scenes evaluate (a pixel of an opaque scene ends after some
    hundred), 12 operations for the exponent and 8 for the blend."""
    kind = case["kind"]
    if kind == "model":
        n = case["rows"]
        return dict(bytes=n * 4 * (8 + 1 + 1) + 3 * 4 * 1377, flops=n * 2 * 1377 * 4)
    if kind == "views":
        n, pix = case["faint"] + 3000 * case["blobs"], case["views"] * case["width"] * case["height"]
        return dict(bytes=n * 40 + pix * 20, flops=pix * 20 * 300)
    pix, P, K = case["width"] * case["height"], case["P"], (case["sh"] + 1) ** 2
    pairs = pix * min(150.0, 60.0 + 40.0 * P / pix)
    if kind == "sort":
        return dict(bytes=P * (8 + 4 + 4) + 4 * 2 * P + pix / 256 * 8, flops=0)
    if kind == "frame":
        return dict(bytes=P * (44 + 12 * K) + pix * 20, flops=P * (250 + 6 * K) + pairs * 20)
    if kind == "train":
        return dict(bytes=P * 2 * (44 + 12 * K) + pix * 44, flops=3 * (P * (250 + 6 * K) + pairs * 20))
    return dict(bytes=P * 2 * 36 + pix * (16 + 12), flops=3 * pairs * 20)


# ---------------------------------------------------------------- the same in 64 bits

def _project64(cam, s, opacity_radius):
    """Eq. 2 for float64 parameters: mean2d, conic, depth, radius (0: culled), colour."""
    f = lambda v: torch.as_tensor(np.asarray(v, np.float64), device=DEV).to(torch.float32).double()  # noqa: E731
    vm = f(cam["viewmat"]).reshape(3, 4)
    R, fx, fy = vm[:, :3], float(cam["fx"]), float(cam["fy"])
    t = s["means3"] @ R.T + vm[:, 3]
    z = t[:, 2]
    front = z > cam["near_z"]
    zs = torch.where(front, z, torch.ones_like(z))
    q = s["quats"] / s["quats"].norm(dim=1, keepdim=True)
    w, x, y, k = q.unbind(1)
    rot = torch.stack([1 - 2 * (y * y + k * k), 2 * (x * y - w * k), 2 * (x * k + w * y), 2 * (x * y + w * k),
                       1 - 2 * (x * x + k * k), 2 * (y * k - w * x), 2 * (x * k - w * y), 2 * (y * k + w * x),
                       1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)
    M = rot * s["scales"][:, None, :]
    limx, limy = 1.3 * 0.5 * cam["width"] / fx, 1.3 * 0.5 * cam["height"] / fy
    xc, yc = (t[:, 0] / zs).clamp(-limx, limx) * zs, (t[:, 1] / zs).clamp(-limy, limy) * zs
    zero = torch.zeros_like(zs)
    J = torch.stack([fx / zs, zero, -fx * xc / zs ** 2, zero, fy / zs, -fy * yc / zs ** 2], 1).reshape(-1, 2, 3)
    A = (J @ R) @ M
    cov = A @ A.transpose(1, 2)
    a, b, c = cov[:, 0, 0] + 0.3, cov[:, 0, 1], cov[:, 1, 1] + 0.3
    det = a * c - b * b
    mean2d = torch.stack([fx * t[:, 0] / zs + cam["cx"], fy * t[:, 1] / zs + cam["cy"]], 1)
    conic = torch.stack([c, -b, a], 1) / det[:, None]
    with torch.no_grad():
        reach2 = 2 * torch.log(255 * s["opacity"]) if opacity_radius else torch.full_like(det, 9.0)
        mid = 0.5 * (a + c)
        lam = mid + (mid * mid - det).clamp_min(0.1).sqrt()
        radius = (reach2.clamp_min(0.0) * lam).sqrt().ceil()
        radius = torch.where(front & (det > 0) & (reach2 > 0), radius, torch.zeros_like(radius))
    d = s["means3"] - f(cam["campos"])
    x, y, k = (d / d.norm(dim=1, keepdim=True)).unbind(1)
    Y = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    deg = s["sh_degree"]
    if deg > 0:
        c1 = math.sqrt(3 / (4 * math.pi))
        Y += [-c1 * y, c1 * k, -c1 * x]
    if deg > 1:
        c2 = 0.5 * math.sqrt(15 / math.pi)
        Y += [c2 * x * y, -c2 * y * k, 0.25 * math.sqrt(5 / math.pi) * (2 * k * k - x * x - y * y), -c2 * x * k,
              0.5 * c2 * (x * x - y * y)]
    if deg > 2:
        c3, c4, c5 = (0.25 * math.sqrt(v / math.pi) for v in (17.5, 10.5, 105.0))
        Y += [-c3 * y * (3 * x * x - y * y), 2 * c5 * x * y * k, -c4 * y * (4 * k * k - x * x - y * y),
              0.25 * math.sqrt(7 / math.pi) * k * (2 * k * k - 3 * x * x - 3 * y * y), -c4 * x * (4 * k * k - x * x - y * y),
              c5 * k * (x * x - y * y), -c3 * x * (x * x - 3 * y * y)]
    rgb = ((torch.stack(Y, 1)[:, :, None] * s["sh"]).sum(1) + 0.5).clamp_min(0.0)
    return mean2d, conic, z, radius, rgb


def _lists64(cam, mean2d, depth, radius):
    """Every tile's Gaussians in depth order: ids, and each tile's first index and length."""
    gw, gh = (cam["width"] + 15) // 16, (cam["height"] + 15) // 16
    lo = ((mean2d - radius[:, None]) / 16).floor().clamp_min(0).long()
    hi = ((mean2d + radius[:, None]) / 16).floor().long()
    hi = torch.minimum(hi, torch.tensor([gw - 1, gh - 1], device=DEV))
    size = (hi - lo + 1).clamp_min(0)
    count = torch.where(radius > 0, size[:, 0] * size[:, 1], torch.zeros_like(size[:, 0]))
    order = torch.sort(depth.float(), stable=True)[1]      # the order is the float32 depths'
    order = order[count[order] > 0]
    n = count[order]
    ids = torch.repeat_interleave(order, n)
    k = torch.arange(ids.numel(), device=DEV) - torch.repeat_interleave(n.cumsum(0) - n, n)
    w = size[ids, 0]
    tile = (lo[ids, 1] + k // w) * gw + lo[ids, 0] + k % w
    tile, at = torch.sort(tile.to(torch.int32), stable=True)
    length = torch.bincount(tile, minlength=gw * gh)
    return ids[at], length.cumsum(0) - length, length


def _pixels(cam, tiles):
    gw = (cam["width"] + 15) // 16
    k = torch.arange(256, device=DEV)
    px = (tiles % gw * 16)[:, None] + k % 16
    py = (tiles // gw * 16)[:, None] + k // 16
    return px, py, (px < cam["width"]) & (py < cam["height"])


def _alpha64(p, ids, px, py, listed_, alpha_max=0.99):
    """alpha of [tiles, 256 pixels, entries], 0 where culled."""
    mean2d, conic, opacity = p
    dx = mean2d[ids, 0][:, None, :] - (px.double() + 0.5)[:, :, None]
    dy = mean2d[ids, 1][:, None, :] - (py.double() + 0.5)[:, :, None]
    s = conic[ids][:, None]
    power = -0.5 * (s[..., 0] * dx * dx + s[..., 2] * dy * dy) - s[..., 1] * dx * dy
    a = (opacity[ids][:, None] * power.exp()).clamp_max(alpha_max)
    return torch.where((a >= 1.0 / 255.0) & listed_[:, None, :], a, torch.zeros_like(a))


def _needed64(cam, p, ids, first, length, step=128):
    """List entries of each tile until all of its pixels have ended."""
    need = torch.zeros_like(length)
    left = torch.nonzero(length > 0).flatten()
    T = torch.ones(length.numel(), 256, dtype=torch.float64, device=DEV)
    at = 0
    while left.numel():
        keep = []
        for part in left.split(512):
            k = at + torch.arange(step, device=DEV)
            ok = k[None] < length[part][:, None]
            g = ids[(first[part][:, None] + k).clamp_max(ids.numel() - 1)]
            px, py, inside = _pixels(cam, part)
            Tn = T[part][:, :, None] * (1 - _alpha64(p, g, px, py, ok)).cumprod(2)
            T[part] = Tn[:, :, -1]
            need[part] = torch.minimum(length[part], torch.full_like(part, at + step))
            going = ((Tn[:, :, -1] >= 1e-4) & inside).any(1) & (length[part] > at + step)
            keep.append(part[going])
        left = torch.cat(keep)
        at += step
    return need


def _blend64(cam, mean2d, conic, opacity, rgb, ids, first, length, dimg=None):
    """Image and transmittance (black background); with dimg (a function of the image), also the
    derivatives with respect to mean2d, conic, opacity and rgb."""
    p = [v.detach() for v in (mean2d, conic, opacity, rgb)]
    with torch.no_grad():
        need = _needed64(cam, p[:3], ids, first, length)
    img = torch.zeros(3, cam["height"], cam["width"], dtype=torch.float64, device=DEV)
    Tf = torch.ones(cam["height"], cam["width"], dtype=torch.float64, device=DEV)
    grads = None

    def groups():
        order = torch.sort(need, descending=True)[1]
        order = order[need[order] > 0]
        sizes = need[order].tolist()
        i = 0
        while i < len(sizes):
            n = max(1, min(len(sizes) - i, 20_000_000 // (256 * sizes[i])))
            yield order[i:i + n], sizes[i]
            i += n

    def tiles_of(part, L, v):
        k = torch.arange(L, device=DEV)
        g = ids[(first[part][:, None] + k).clamp_max(ids.numel() - 1)]
        px, py, inside = _pixels(cam, part)
        a = _alpha64(v[:3], g, px, py, k[None] < need[part][:, None])
        with torch.no_grad():
            alive = (1 - a).cumprod(2) >= 1e-4        # false from the fragment that ends the pixel on
        a = torch.where(alive, a, torch.zeros_like(a))
        after = (1 - a).cumprod(2)
        w = a * torch.cat([torch.ones_like(after[:, :, :1]), after[:, :, :-1]], 2)
        return torch.bmm(w, v[3][g]), after[:, :, -1], px, py, inside

    with torch.no_grad():
        for part, L in groups():
            c, t, px, py, inside = tiles_of(part, L, p)
            img[:, py[inside], px[inside]] = c[inside].T
            Tf[py[inside], px[inside]] = t[inside]
    if dimg is not None:
        G = dimg(img)
        grads = [torch.zeros_like(v) for v in p]
        for part, L in groups():
            leaf = [v.clone().requires_grad_(True) for v in p]
            c, _, px, py, inside = tiles_of(part, L, leaf)
            (c[inside] * G[:, py[inside], px[inside]].T).sum().backward()
            for s, v in zip(grads, leaf):
                s += v.grad
    return img, Tf, grads


def _frame64(cam, scene, tight):
    s = {k: (v.double() if isinstance(v, torch.Tensor) else v) for k, v in scene.items()}
    mean2d, conic, depth, radius, rgb = _project64(cam, s, tight)
    ids, first, length = _lists64(cam, mean2d, depth, radius)
    img, T, _ = _blend64(cam, mean2d, conic, s["opacity"], rgb, ids, first, length)
    return img, T


def _model64(state):
    """The cost model with its FP16 roundings (weights, input, hidden activations), sums in 64 bits."""
    r16 = lambda v: v.float().half().double()  # noqa: E731
    P = state["model"].params
    cut = [0, 256, 288, 1312, 1344, 1376, 1377]
    w = [r16(P[a:b]).requires_grad_(True) for a, b in zip(cut, cut[1:])]
    through = lambda v: v + (r16(v) - v).detach()  # noqa: E731
    x = r16((state["x"] - state["norm"][:8]) * state["norm"][8:])
    h = through((x @ w[0].reshape(32, 8).T + w[1]).relu())
    h = through((h @ w[2].reshape(32, 32).T + w[3]).relu())
    y = h @ w[4] + w[5]
    loss = ((y - state["y"].double()) ** 2).mean()
    loss.backward()
    return dict(cost=y.detach(), grad=torch.cat([v.grad for v in w]), loss=loss.detach().reshape(1))


def exact(case, seed):
    kind = case["kind"]
    if kind == "sort" or case.get("scene") == "box_cluster":
        return None      # whole numbers only; 1.3 billion list entries
    if kind == "model":
        return _model64(prepare(case, seed))
    if kind == "views":
        cams, scene = _occluded(case, seed)
        found = [_frame64(cam, scene, False) for cam in cams]
        return [dict(img=i, T_final=t, n_contrib=None) for i, t in found]
    if kind == "frame":
        cam, scene = _scene(case, seed)
        img, T = _frame64(cam, scene, bool(case.get("tight")))
        return dict(img=img, T_final=T, n_contrib=None, n_splats=None)
    if kind == "blend":
        state = prepare(case, seed)      # its inputs are float32 values of the projection
        p = {k: v.detach().double() for k, v in state["leaves"].items()}
        r = state["bins"]["tile_ranges"].long() & 0xFFFFFFFF
        ids = state["bins"]["ids_sorted"].long()
        weight = state["weight"].double()
        img, T, g = _blend64(state["cam"], p["mean2d"], p["conic"], p["opacity"], p["rgb"], ids, r[:, 0], r[:, 1] - r[:, 0],
                             lambda _: weight)
        return dict(img=img, T=T, dmean2d=g[0], dconic=g[1], dopacity=g[2], drgb=g[3])
    cam, scene = _scene(case, seed)
    target = _target(case, seed).double()
    s = {k: (v.double().requires_grad_(True) if isinstance(v, torch.Tensor) else v) for k, v in scene.items()}
    mean2d, conic, depth, radius, rgb = _project64(cam, s, False)
    ids, first, length = _lists64(cam, mean2d.detach(), depth.detach(), radius)
    img, T, g = _blend64(cam, mean2d, conic, s["opacity"], rgb, ids, first, length,
                         lambda i: (i - target).sign() / i.numel())
    used = radius > 0
    torch.autograd.backward([mean2d, conic, rgb], [torch.where(used[:, None], v, torch.zeros_like(v)) for v in (g[0], g[1], g[3])])
    zero = lambda v: v if v is not None else 0  # noqa: E731
    return dict(img=img, T=T, **{"d" + k: zero(s[k].grad) + (g[2] if k == "opacity" else 0)
                                 for k in ("means3", "scales", "quats", "opacity", "sh")})
