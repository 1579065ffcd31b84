"""The work that a user of this rasterizer has it do, as measurable cases.

A case names a path (its "op") and its sizes and options:

  forward    Rasterizer.forward: projection, per-tile lists, compositing of one view
  autograd   DarbRasterize in a torch graph: forward and backward to the splat attributes
  train      one fused training step: projection, lists, compositing with the L1 loss,
             compositing backward, chain rule + Adam
  project    darb_preprocess alone
  sort       darb_bin_sort alone (asynchronous capacity mode, as in a training loop)
  composite  darb_render_fwd alone
  composite_bwd  darb_render_bwd alone
  chain_adam darb_preprocess_bwd and darb_adam_step: the unfused tail of a data-parallel step
  dssim      darb_l1_dssim_loss: the full image loss and its gradient
  density    darb_densify_stats and darb_densify: one round of adaptive density control
  batch      BatchRenderer.replay: many cameras of one scene in one captured batch

Scenes are the clustered and the uniform scene of paper_2501_12369_gb300.synth, drawn on the GPU.
exact() gives what run() returns in 64 bits, from the definition of the method, in plain torch.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

from paper_2501_12369_gb300 import darb, synth

DEV = "cuda"
KERNELS = ("gaussian", "half_cosine", "raised_cosine", "mod_sinc", "inv_quadric", "inv_multiquadric", "parabola")
# A modified member of the kernel family: cos(d_M^1.5 / 3), with a psi set by hand.
MODIFIED = dict(base="half_cosine", xi=3.0, beta=1.5, psi=1.3)
# psi, q_max and whether the limit is strict, as the paper prints them (the modified member: xi, beta above).
PSI = dict(gaussian=1.0, half_cosine=1.36, raised_cosine=0.655, mod_sinc=1.18, inv_quadric=1.38,
           inv_multiquadric=1.61, parabola=1.3, modified=1.3)
QMAX = dict(raised_cosine=6.25, modified=min(9.0, (3.0 * math.pi / 2) ** (2 / 1.5)))
STRICT = ("inv_quadric", "inv_multiquadric")
# Learning rates of a run's last phase (the 3DGS rates at the end of their decay), so that a state that is
# stepped many times stays the scene it was.
LRS = (9.6e-6, 5e-5, 1e-5, 2e-4, 2.5e-5, 1.25e-6)
BETA1, BETA2, EPS, STEP = 0.9, 0.999, 1e-15, 20000
LAMBDA = 0.2
DENSIFY = dict(grad_threshold=0.0002, dense_scale=0.06, min_opacity=0.05, max_screen_radius=600.0,
               max_world_scale=0.12, split_scale_div=1.6)


# ---------------------------------------------------------------------------- the cases

def listed():
    return [
        # The smallest call: a handful of splats in a thumbnail, where launches are the time (a
        # program that optimises a toy scene, or a preview).
        dict(name="forward_1k_thumbnail", op="forward", n=1024, width=64, height=64, tile=16, kernel="half_cosine", sh=0),
        # A small scene in a torch training loop with other losses than the built-in ones; the image
        # is no multiple of any tile.
        dict(name="autograd_20k_ragged", op="autograd", n=20000, width=333, height=207, tile=16, kernel="gaussian", sh=3),
        # Viewing one camera of a medium scene at 720p, by the default calls.
        dict(name="forward_500k_720p", op="forward", n=500000, width=1280, height=720, tile=16, kernel="half_cosine", sh=3),
        # The headline: a training step of a full-size scene at 1080p.
        dict(name="train_3m_1080p", op="train", n=3000000, width=1920, height=1080, tile=32, kernel="half_cosine", sh=3),
        # Projection alone, as every view begins.
        dict(name="project_1m_1080p", op="project", n=1000000, width=1920, height=1080, tile=32, kernel="half_cosine", sh=3),
        # The per-tile lists alone, with the tiles that 3DGS uses.
        dict(name="sort_1m_1080p_tile16", op="sort", n=1000000, width=1920, height=1080, tile=16, kernel="half_cosine",
             sh=0, keys=False),
        # Compositing of the plain Gaussian, whose pixels walk the longest lists.
        dict(name="composite_gaussian_1m_1080p", op="composite", n=1000000, width=1920, height=1080, tile=32,
             kernel="gaussian", sh=0),
        # Its backward, for a kernel with a costly derivative, on 16-pixel tiles and an odd image.
        dict(name="composite_bwd_sinc_300k", op="composite_bwd", n=300000, width=1245, height=825, tile=16,
             kernel="mod_sinc", sh=0),
        # The tail of a step whose gradients are reduced over ranks between the two calls.
        dict(name="chain_adam_1m_odd", op="chain_adam", n=1000003, width=1920, height=1080, tile=16, kernel="half_cosine", sh=3),
        # The paper's full image loss at 1080p.
        dict(name="dssim_1080p", op="dssim", width=1920, height=1080),
        # Density control of a medium training state, as it runs every hundred steps.
        dict(name="density_1m", op="density", n=1000000, width=1920, height=1080, sh=3),
        # A camera path or a server's full batch: mixed resolutions in one captured batch.
        dict(name="batch_16_views_1m", op="batch", n=1000000, views=16, tile=32, kernel="half_cosine", sh=3, scale=1.0),
    ]


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    def span(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def image(lo, hi):
        w = span(lo, hi)
        return dict(width=w, height=max(40, int(w * rng.uniform(0.5, 1.0)) if w < 1000 else int(w * rng.uniform(0.5, 0.65))))

    op = rng.choice(("forward", "autograd", "train", "project", "sort", "composite", "composite_bwd", "chain_adam",
                     "dssim", "density", "batch"))
    kernel = rng.choice(KERNELS)
    sh = rng.choice((0, 1, 2, 3, 3, 3))
    tile = rng.choice((8, 16, 16, 32, 32))
    if op == "forward":
        return dict(op=op, n=span(500, 1000000), tile=tile, kernel=kernel, sh=sh, **image(64, 1920))
    if op == "autograd":
        return dict(op=op, n=span(2000, 500000), tile=tile, kernel=kernel, sh=sh, **image(100, 1280))
    if op == "train":
        return dict(op=op, n=span(50000, 3000000), tile=rng.choice((16, 32)), kernel="half_cosine", sh=rng.choice((1, 2, 3)),
                    **image(480, 1920))
    if op == "project":
        return dict(op=op, n=span(5000, 3000000), tile=tile, kernel=kernel, sh=sh, **image(320, 1920))
    if op == "sort":
        return dict(op=op, n=span(2000, 3000000), tile=tile, kernel=kernel, sh=0, keys=rng.random() < 0.2, **image(128, 1920))
    if op in ("composite", "composite_bwd"):
        return dict(op=op, n=span(5000, 1000000), tile=tile, kernel=rng.choice(KERNELS + ("modified",)), sh=0,
                    **image(128, 1920))
    if op == "chain_adam":
        return dict(op=op, n=span(5000, 2000000), tile=16, kernel=kernel, sh=sh, **image(320, 1920))
    if op == "dssim":
        return dict(op=op, **image(100, 2560))
    if op == "density":
        return dict(op=op, n=span(5000, 1500000), sh=sh, **image(320, 1920))
    return dict(op=op, n=span(20000, 1000000), views=rng.randint(1, 16), tile=rng.choice((16, 32)), kernel=kernel, sh=sh,
                scale=round(rng.uniform(0.4, 1.0), 3))


# ---------------------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)


def _scene(case, seed):
    """The uniform cube for the smallest scenes, else the clustered scene: means, scales, quats, opacities, sh."""
    g = _generator(seed)
    n, k = case["n"], (case["sh"] + 1) ** 2

    def rand(*s):
        return torch.rand(*s, generator=g, device=DEV)

    def randn(*s):
        return torch.randn(*s, generator=g, device=DEV)

    if n < 2000:
        means, lo, hi = rand(n, 3) * 2 - 1, -4.0, -2.0
    else:
        centres, sig = rand(20, 3) * 10 - 5, rand(20, 3) * 1.2 + 0.3
        rots = torch.linalg.qr(randn(20, 3, 3))[0]
        which = torch.randint(0, 20, (n,), generator=g, device=DEV)
        z = randn(n, 3) * sig[which]
        means = (centres[which] + (rots[which] * z[:, None, :]).sum(-1)).clamp(-5.0, 5.0)
        lo, hi = -5.0, -2.0
    scales = torch.exp(rand(n, 3) * (hi - lo) + lo)
    quats = randn(n, 4)
    quats = quats / quats.norm(dim=1, keepdim=True)
    opac = torch.sigmoid(randn(n))
    sh = torch.randn(n, k, 3, generator=g, device=DEV) * 0.2
    sh[:, 0] = (rand(n, 3) * 2 - 1) * synth.DC_HALF_RANGE
    return darb.SplatTensors(*(t.float().contiguous() for t in (means, scales, quats, opac, sh)), case["sh"]), g


def _camera(case, seed):
    w, h = case["width"], case["height"]
    if case["n"] < 2000:
        return synth.pinhole((0.0, 0.3 * math.sin(seed), 4.0), w, h, float(w))
    return synth.fibonacci_cameras(100, 6.0, w, h, 1500.0 / 1920.0 * w)[int(seed) % 100]


def _cameras(case, seed):
    """Random poses; the three resolutions in turn, so that every seed renders as many pixels."""
    rng, cams = np.random.default_rng(int(seed) + 1), []
    for i in range(case["views"]):
        w, h = (max(64, int(v * case["scale"])) for v in synth.MULTIVIEW_RESOLUTIONS[(i + 2) % 3])
        v = rng.normal(size=3)
        cams.append(synth.pinhole(5.0 * v / np.linalg.norm(v), w, h, 1500.0 / 1920.0 * w))
    return cams


def _kparams(kernel):
    if kernel == "modified":
        return darb.darb_kernel_generic(MODIFIED["base"], MODIFIED["xi"], MODIFIED["beta"], 1, MODIFIED["psi"])
    return darb.darb_kernel_defaults(kernel)


def _projected(n):
    """Projected records that start as zeros: a culled splat's record is only partly written."""
    p = darb.Projected.empty(n, DEV)
    for f in ("depth", "radius", "tile_rect", "mean2d", "conic_o", "rgb", "clamped", "tiles_touched", "tile_runs"):
        getattr(p, f).zero_()
    return p


def _lists(s, splats, cam, tile, kp, keys=False, slack=1.3):
    """The projected records and buffers for the lists of one view, sized by a counting pass."""
    n = splats.n
    s.proj = darb.darb_preprocess(splats, cam, kp, tile, _projected(n))
    cap = 1024
    while True:
        tx, ty = darb.darb_tile_grid(cam, tile)
        ws = torch.empty(darb.darb_bin_sort_workspace_size(n, tile, cam, cap), dtype=torch.uint8, device=DEV)
        bins = darb.Binning.empty(cap, tx * ty, DEV, keys=keys)
        try:
            m = darb.darb_bin_sort(s.proj, n, tile, cam, ws, cap, bins).M
        except darb.DarbError as e:
            cap = int(e.M * slack) + 1024
            continue
        s.ws, s.bins, s.cap, s.m = ws, bins, cap, m
        return


def _image(cam):
    return darb.ImageOut(*(t.zero_() for t in (torch.empty(3, cam.height, cam.width, device=DEV),
                                               torch.empty(cam.height, cam.width, device=DEV),
                                               torch.empty(cam.height, cam.width, dtype=torch.int32, device=DEV),
                                               torch.empty(cam.height, cam.width, dtype=torch.int32, device=DEV))))


def _training(splats, g):
    """Raw parameters and the moments of a run that has been going for a while."""
    p = types.SimpleNamespace(means=splats.means, log_scales=torch.log(splats.scales), quats=splats.quats,
                              opacity_logits=torch.logit(splats.opacities), sh=splats.sh, scales=splats.scales,
                              opacities=splats.opacities, sh_degree=splats.sh_degree)
    st = types.SimpleNamespace()
    for f, like in (("means", p.means), ("scales", p.means), ("quats", p.quats), ("opac", p.opacities), ("sh", p.sh)):
        setattr(st, "m_" + f, torch.randn(like.shape, generator=g, device=DEV) * 1e-6)
        setattr(st, "v_" + f, (torch.rand(like.shape, generator=g, device=DEV) * 1.5 + 0.5) * 1e-12)
    return p, st


MOMENTS = tuple(m + f for f in ("means", "scales", "quats", "opac", "sh") for m in ("m_", "v_"))
PARAMS = ("means", "log_scales", "quats", "opacity_logits", "sh", "scales", "opacities")


def prepare(case, seed):
    op = case["op"]
    s = types.SimpleNamespace(case=case, op=op)
    if op == "dssim":
        g = _generator(seed)
        s.target = torch.rand(3, case["height"], case["width"], generator=g, device=DEV)
        s.image = (0.7 * s.target + 0.3 * torch.rand(s.target.shape, generator=g, device=DEV)).contiguous()
        s.ws = torch.empty(darb.darb_l1_dssim_workspace_size(case["width"], case["height"]), dtype=torch.uint8, device=DEV)
        s.dl, s.loss = torch.zeros_like(s.image), torch.zeros(2, device=DEV)
        return s
    s.splats, g = _scene(case, seed)
    n = s.splats.n
    if op == "density":
        s.params, s.state = _training(s.splats, g)
        s.grad2d = torch.randn(n, 12, generator=g, device=DEV) * 2e-7
        visible = torch.rand(n, generator=g, device=DEV) < 0.4
        s.radius = torch.where(visible, torch.randint(1, 700, (n,), generator=g, device=DEV), 0).int()
        s.count = torch.randint(0, 60, (n,), generator=g, device=DEV).float()
        s.accum = s.count * torch.rand(n, generator=g, device=DEV) * 0.00025
        s.max_radius = torch.randint(0, 620, (n,), generator=g, device=DEV).int()
        s.normals = torch.randn(n, 2, 3, generator=g, device=DEV)
        s.cfg = darb.darb_densify_cfg(*(DENSIFY[f] for f, _ in darb.darb_densify_cfg._fields_))
        grown = {f: torch.zeros((2 * n,) + tuple(getattr(s.params, f).shape[1:]), device=DEV) for f in PARAMS}
        s.out = types.SimpleNamespace(**grown, sh_degree=case["sh"])
        s.out_state = types.SimpleNamespace(**{f: torch.zeros((2 * n,) + tuple(getattr(s.state, f).shape[1:]), device=DEV)
                                               for f in MOMENTS})
        return s
    if op == "batch":
        s.views = darb.BatchRenderer(s.splats, _cameras(case, seed), case["kernel"], case["tile"], 8)
        s.views.capture()
        return s
    s.cam, s.tile, s.kp = _camera(case, seed), case["tile"], _kparams(case["kernel"])
    w, h = s.cam.width, s.cam.height
    if op in ("forward", "autograd"):
        s.rast = darb.Rasterizer(s.cam, s.kp, s.tile)
        if op == "autograd":
            s.leaves = [t.clone().requires_grad_(True) for t in (s.splats.means, s.splats.scales, s.splats.quats,
                                                                 s.splats.opacities, s.splats.sh)]
            s.dl = torch.rand(3, h, w, generator=g, device=DEV) * 2 - 1
        return s
    if op == "project":
        s.proj = _projected(n)
        return s
    if op == "chain_adam":
        s.params, s.state = _training(s.splats, g)
        s.proj = darb.darb_preprocess(s.splats, s.cam, s.kp, s.tile, _projected(n))
        s.grad2d = torch.randn(n, 12, generator=g, device=DEV) * 1e-6
        s.grad2d[:, 9:] = 0
        s.grad2d[~_inside(s.splats, s.cam)] = 0  # splats that no pixel reached have no gradient
        s.grads = darb.SplatGrads.empty_flat(n, case["sh"], DEV)
        s.cfg = darb.darb_adam_config(*LRS, BETA1, BETA2, EPS, STEP)
        return s
    _lists(s, s.splats, s.cam, s.tile, s.kp, keys=case.get("keys", False))
    if op == "sort":
        # buffers of one size for every seed, zero past the instances; the capacity in use stays s.cap
        size = {8: 64, 16: 24, 32: 12}[s.tile] * n + 65536
        s.cap = min(s.cap, size)
        s.bins.values = torch.zeros(size, dtype=torch.int32, device=DEV)
        if s.bins.keys is not None:
            s.bins.keys = torch.zeros(size, dtype=torch.int64, device=DEV)
        return s
    s.img = _image(s.cam)
    if op == "composite_bwd":
        darb.darb_render_fwd(s.proj, s.bins, s.cam, s.kp, s.tile, s.img)
        s.dl = (torch.rand(3, h, w, generator=g, device=DEV) * 2 - 1) / (3 * w * h)
        s.grad2d = torch.zeros(n, 12, device=DEV)
    if op == "train":
        s.params, s.state = _training(s.splats, g)
        s.target = torch.rand(3, h, w, generator=g, device=DEV)
        s.img = darb.ImageOut(None, s.img.t_final, s.img.last, None)  # a step needs no image, only its loss
        s.dl, s.loss = torch.zeros(3, h, w, device=DEV), torch.zeros(1, device=DEV)
        s.grad2d = torch.zeros(n, 12, device=DEV)
        s.cfg = darb.darb_adam_config(*LRS, BETA1, BETA2, EPS, STEP)
    return s


# ---------------------------------------------------------------------------- one pass

def run(s):
    op = s.op
    if op == "forward":
        proj, bins, img = s.rast.forward(s.splats)
        return dict(image=img.image, t_final=img.t_final, last=img.last, n_contrib=img.n_contrib, ranges=bins.ranges,
                    num=bins.num_instances, radius=proj.radius)
    if op == "autograd":
        for t in s.leaves:
            t.grad = None
        image = darb.DarbRasterize.apply(*s.leaves, s.splats.sh_degree, s.rast)
        image.backward(s.dl)
        return dict(image=image.detach(), **{k: t.grad for k, t in zip(("means", "scales", "quats", "opacities", "sh"), s.leaves)})
    if op == "dssim":
        darb.darb_l1_dssim_loss(s.image, s.target, LAMBDA, s.ws, s.dl, s.loss)
        return dict(grad=s.dl, loss=s.loss)
    if op == "density":
        w, h = s.case["width"], s.case["height"]
        darb.darb_densify_stats(s.grad2d, s.radius, w, h, s.accum, s.count, s.max_radius)
        n_out = darb.darb_densify(s.params, s.state, s.accum, s.count, s.max_radius, s.normals, s.cfg, s.out, s.out_state)
        return dict(n_out=n_out, accum=s.accum, count=s.count, max_radius=s.max_radius,
                    **{f: getattr(s.out, f) for f in PARAMS}, **{f: getattr(s.out_state, f) for f in MOMENTS})
    if op == "batch":
        s.views.replay()
        return dict(images=[o.image for o in s.views.outs], num=s.views.num_instances, status=s.views.status)
    n, cam, kp, tile = s.splats.n, s.cam, s.kp, s.tile
    if op == "project":
        p = darb.darb_preprocess(s.splats, cam, kp, tile, s.proj)
        return dict(depth=p.depth, mean2d=p.mean2d, conic_o=p.conic_o, rgb=p.rgb, radius=p.radius, tile_rect=p.tile_rect,
                    tiles_touched=p.tiles_touched, tile_runs=p.tile_runs, clamped=p.clamped)
    if op == "sort":
        b = darb.darb_bin_sort(s.proj, n, tile, cam, s.ws, s.cap, s.bins, sync=False)
        out = dict(values=b.values, ranges=b.ranges, num=b.num_instances, status=b.status)
        return dict(out, keys=b.keys) if b.keys is not None else out
    if op == "composite":
        o = darb.darb_render_fwd(s.proj, s.bins, cam, kp, tile, s.img)
        return dict(image=o.image, t_final=o.t_final, last=o.last, n_contrib=o.n_contrib)
    if op == "composite_bwd":
        return dict(grad2d=darb.darb_render_bwd(s.proj, n, s.bins, cam, kp, tile, s.img, s.dl, s.grad2d))
    if op == "chain_adam":
        g = darb.darb_preprocess_bwd(s.splats, cam, kp, s.proj, s.grad2d, s.grads)
        darb.darb_adam_step(s.params, g, s.state, s.cfg)
        return dict(dmeans=g.dmeans, dscales=g.dscales, dquats=g.dquats, dopacities=g.dopacities, dsh=g.dsh,
                    **{f: getattr(s.params, f) for f in PARAMS}, **{f: getattr(s.state, f) for f in MOMENTS})
    darb.darb_preprocess(s.splats, cam, kp, tile, s.proj)
    darb.darb_bin_sort(s.proj, n, tile, cam, s.ws, s.cap, s.bins, sync=False)
    darb.darb_render_fwd_l1(s.proj, s.bins, cam, kp, tile, s.target, s.img, s.dl, s.loss)
    darb.darb_render_bwd(s.proj, n, s.bins, cam, kp, tile, s.img, s.dl, s.grad2d)
    darb.darb_preprocess_bwd_adam(s.params, cam, kp, s.proj, s.grad2d, s.state, s.cfg)
    return dict(loss=s.loss, **{f: getattr(s.params, f) for f in PARAMS}, **{f: getattr(s.state, f) for f in MOMENTS})


# ---------------------------------------------------------------------------- what a pass cannot do without

VISIBLE = 0.4      # of a clustered scene's splats, seen from one of its cameras
PER_TILE = {8: 26, 16: 12, 32: 6}  # member tiles of a visible splat at 1080p
# (pixel, splat) pairs of a pixel up to the last one that it blends, by kernel, in the clustered scenes
PAIRS = dict(gaussian=91, half_cosine=21, raised_cosine=77, mod_sinc=41, inv_quadric=74, inv_multiquadric=34,
             parabola=32, modified=28)
FLOPS_FWD, FLOPS_BWD = 30, 75  # of a pair
RECORD = 4 + 4 + 16 + 8 + 16 + 12 + 1 + 4 + 8


def work(case):
    op = case["op"]
    px = case.get("width", 0) * case.get("height", 0)
    if op == "dssim":
        return dict(bytes=36 * px, flops=3 * px * 2 * (8 * 11 * 2 + 40))
    n, k3 = case["n"], 3 * (case["sh"] + 1) ** 2
    per = 11 + k3
    if op == "density":  # every parameter and moment read and written, with the statistics
        return dict(bytes=n * (4 * (3 * per + 4) * 2 + 24 + 40), flops=n * 40)
    if op == "batch":
        px = int(case["views"] * 1.1e6 * case["scale"] ** 2)
    pairs = px * PAIRS[case["kernel"]] * min(1.0, n / 2e5)
    views = case.get("views", 1)
    vis = n if n < 2000 else int(VISIBLE * n)
    m = vis * max(1.0, PER_TILE[case["tile"]] * max(0.1, min(1.0, px / views / 2.07e6)))
    project = n * 40 + vis * (4 + 4 * k3 + RECORD)
    sort = n * 8 + vis * 28 + m * 4
    walked = min(pairs / 64, m) * 44
    composite = walked + px * 24
    if op == "project":
        return dict(bytes=project, flops=n * 250 + vis * 2 * 4 * k3)
    if op == "sort":
        return dict(bytes=sort + (m * 8 if case["keys"] else 0), flops=0)
    if op == "composite":
        return dict(bytes=composite, flops=pairs * FLOPS_FWD)
    if op == "composite_bwd":
        return dict(bytes=walked + px * 20 + n * 48, flops=pairs * FLOPS_BWD)
    if op == "chain_adam":  # gradients written and read once, every parameter and moment read and written
        return dict(bytes=n * (4 * per * 2 + 24 * per + 32 + 4) + vis * 49, flops=n * 15 * per + vis * 600)
    if op == "forward":
        return dict(bytes=project + sort + m * 4 + composite, flops=n * 250 + pairs * FLOPS_FWD)
    if op == "batch":
        return dict(bytes=n * (44 + 4 * k3) + views * (vis * RECORD + vis * 28 + m * 4) + walked + px * 12,
                    flops=views * n * 250 + pairs * FLOPS_FWD)
    if op == "autograd":
        return dict(bytes=project + sort + m * 4 + composite + px * 20 + n * 48 + n * 4 * per + vis * (4 * per + 49),
                    flops=n * 250 + vis * 600 + pairs * (FLOPS_FWD + FLOPS_BWD))
    return dict(bytes=project + sort + walked * 2 + px * (12 + 12 + 8 + 20) + n * 48 + n * (24 * per + 32 + 4) + vis * 49,
                flops=n * 250 + vis * 600 + n * 15 * per + pairs * (FLOPS_FWD + FLOPS_BWD))


# ---------------------------------------------------------------------------- the same in 64 bits

def _view64(cam):
    v = torch.tensor(np.asarray(cam.viewmat, np.float32), dtype=torch.float64, device=DEV)
    return v[:3, :3], v[:3, 3]


def _inside(splats, cam):
    """Splats in front of the camera whose centre falls into the image."""
    R, t = _view64(cam)
    p = splats.means.double() @ R.T + t
    x, y = cam.fx * p[:, 0] / p[:, 2] + cam.cx, cam.fy * p[:, 1] / p[:, 2] + cam.cy
    return (p[:, 2] > cam.near + 1e-3) & (x > 1) & (x < cam.width - 1) & (y > 1) & (y < cam.height - 1)


def _project64(means, scales, quats, sh, cam, kernel):
    """Centre, conic, covariance, depth and colour of every splat (Eq. 2x2covProjection, real SH colour)."""
    R, t = _view64(cam)
    p = means @ R.T + t
    q = quats / quats.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                       2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                       2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    m = rot * scales[:, None, :]
    tz = p[:, 2]
    tx, ty = p[:, 0] / tz, p[:, 1] / tz
    lx, ly = 1.3 * cam.width / (2 * cam.fx), 1.3 * cam.height / (2 * cam.fy)
    cx, cy = tx.clamp(-lx, lx), ty.clamp(-ly, ly)
    t0 = (cam.fx / tz)[:, None] * R[0] - (cam.fx * cx / tz)[:, None] * R[2]
    t1 = (cam.fy / tz)[:, None] * R[1] - (cam.fy * cy / tz)[:, None] * R[2]
    a0, a1 = (t0[:, :, None] * m).sum(1), (t1[:, :, None] * m).sum(1)
    psi = float(np.float32(PSI[kernel]))
    a, b, c = psi * (a0 * a0).sum(1) + 0.3, psi * (a0 * a1).sum(1), psi * (a1 * a1).sum(1) + 0.3
    det = a * c - b * b
    d = means + (R.T @ t)
    rgb = (_sh64(d / d.norm(dim=1, keepdim=True), sh.shape[1])[:, :, None] * sh).sum(1) + 0.5
    return types.SimpleNamespace(u=torch.stack([cam.fx * tx + cam.cx, cam.fy * ty + cam.cy], 1),
                                 conic=torch.stack([c / det, -b / det, a / det], 1), cov=(a, b, c, det), depth=tz,
                                 rgb=rgb.clamp(min=0.0))


def _sh64(d, k):
    x, y, z = d.unbind(1)
    xx, yy, zz = x * x, y * y, z * z
    pi = math.pi
    c1, c2 = math.sqrt(3 / (4 * pi)), math.sqrt(15 / (4 * pi))
    c3a, c3c = math.sqrt(35 / (32 * pi)), math.sqrt(21 / (32 * pi))
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if k > 1:
        Y += [-c1 * y, c1 * z, -c1 * x]
    if k > 4:
        Y += [c2 * x * y, -c2 * y * z, math.sqrt(5 / (16 * pi)) * (2 * zz - xx - yy), -c2 * x * z, 0.5 * c2 * (xx - yy)]
    if k > 9:
        Y += [-c3a * y * (3 * xx - yy), math.sqrt(105 / (4 * pi)) * x * y * z, -c3c * y * (4 * zz - xx - yy),
              math.sqrt(7 / (16 * pi)) * z * (2 * zz - 3 * xx - 3 * yy), -c3c * x * (4 * zz - xx - yy),
              math.sqrt(105 / (16 * pi)) * z * (xx - yy), -c3a * x * (xx - 3 * yy)]
    return torch.stack(Y, 1)


def _visible64(p, cam, tile, kernel):
    """Splats that are not culled: in front, with a rectangle in the image and an ellipse that reaches a tile of it."""
    a, b, c, det = p.cov
    W, H = cam.width, cam.height
    mid = 0.5 * (a + c)
    rad = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0))))
    x0, x1 = torch.ceil(p.u[:, 0] - rad - 0.5).clamp(min=0), torch.floor(p.u[:, 0] + rad - 0.5).clamp(max=W - 1)
    y0, y1 = torch.ceil(p.u[:, 1] - rad - 0.5).clamp(min=0), torch.floor(p.u[:, 1] + rad - 0.5).clamp(max=H - 1)
    ok = (p.depth > cam.near) & (x0 <= x1) & (y0 <= y1)
    idx = ok.nonzero()[:, 0]
    A, B, C = p.conic[idx].unbind(1)
    u0, u1 = p.u[idx].unbind(1)
    y0, y1 = y0[idx], y1[idx]
    qm, dt = QMAX.get(kernel, 9.0), A * C - B * B
    xm, ym = torch.sqrt(qm * C / dt), torch.sqrt(qm * A / dt)
    yr = -B * xm / C
    member = torch.zeros_like(A, dtype=torch.bool)
    for r in range(-(-H // tile)):
        ea = torch.maximum(r * tile + 0.5 - u1, -ym)
        eb = torch.minimum(min((r + 1) * tile, H) - 0.5 - u1, ym)
        dr, dl = torch.minimum(torch.maximum(yr, ea), eb), torch.minimum(torch.maximum(-yr, ea), eb)
        right = (-B * dr + torch.sqrt((A * qm - dt * dr * dr).clamp(min=0))) / A
        left = (-B * dl - torch.sqrt((A * qm - dt * dl * dl).clamp(min=0))) / A
        member |= ((ea <= eb) & (y1 >= r * tile) & (y0 < (r + 1) * tile) &
                   (torch.ceil(u0 + left - 0.5).clamp(min=0) <= torch.floor(u0 + right - 0.5).clamp(max=W - 1)))
    keep = torch.zeros_like(ok)
    keep[idx[member]] = True
    return keep


def _profile64(q, kernel):
    if kernel == "gaussian":
        return torch.exp(-0.5 * q)
    if kernel == "half_cosine":
        return torch.cos(q * (math.pi / 18))
    if kernel == "raised_cosine":
        return 0.5 + 0.5 * torch.cos(torch.sqrt(q.clamp(min=1e-300)) * (math.pi / 2.5))
    if kernel == "mod_sinc":
        x = torch.sqrt(q.clamp(min=1e-24)) * (math.pi / 3)
        return torch.sin(x) / x
    if kernel == "inv_quadric":
        return 1 / (1 + q)
    if kernel == "inv_multiquadric":
        return torch.rsqrt(1 + q)
    if kernel == "parabola":
        return 1 - q / 9
    return torch.cos(q.clamp(min=1e-300) ** (MODIFIED["beta"] / 2) / MODIFIED["xi"])


def _composite64(p, opac, cam, kernel, keep, upstream=None):
    """Front-to-back compositing of the kept splats.  upstream(image tile, rows, columns) gives the
    gradient w.r.t. the image; returns image, T and the gradients [n, 12] w.r.t. centre, conic,
    opacity and colour."""
    W, H, qm = cam.width, cam.height, QMAX.get(kernel, 9.0)
    order = keep.nonzero()[:, 0]
    order = order[torch.argsort(p.depth.detach()[order].float(), stable=True)]
    cols = torch.cat([p.u, p.conic, opac[:, None], p.rgb], 1).detach()[order]  # x y A B C o r g b
    dt = cols[:, 2] * cols[:, 4] - cols[:, 3] ** 2
    xm, ym = torch.sqrt(qm * cols[:, 4] / dt), torch.sqrt(qm * cols[:, 2] / dt)
    image = torch.zeros(3, H, W, dtype=torch.float64, device=DEV)
    T = torch.ones(H, W, dtype=torch.float64, device=DEV)
    grad = torch.zeros(p.u.shape[0], 12, dtype=torch.float64, device=DEV) if upstream else None
    bg = torch.tensor([float(b) for b in cam.bg], dtype=torch.float64, device=DEV)
    step = 32
    for y0 in range(0, H, step):
        y1 = min(y0 + step, H)
        row = ((cols[:, 1] + ym > y0) & (cols[:, 1] - ym < y1)).nonzero()[:, 0]
        rx, rm = cols[row, 0], xm[row]
        for x0 in range(0, W, step):
            x1 = min(x0 + step, W)
            own = row[((rx + rm > x0) & (rx - rm < x1)).nonzero()[:, 0]]
            ys, xs = torch.meshgrid(torch.arange(y0, y1, device=DEV) + 0.5, torch.arange(x0, x1, device=DEV) + 0.5, indexing="ij")
            px, py = xs.reshape(-1, 1).double(), ys.reshape(-1, 1).double()
            take = 256
            while True:
                c = cols[own[:take]]
                if upstream:
                    c = c.requires_grad_(True)
                dx, dy = c[:, 0] - px, c[:, 1] - py
                q = c[:, 2] * dx * dx + 2 * c[:, 3] * dx * dy + c[:, 4] * dy * dy
                alpha = (c[:, 5] * _profile64(q, kernel)).clamp(max=0.99)
                inside = (q < qm) if kernel in STRICT else (q <= qm)
                alpha = torch.where(inside & (alpha >= 1 / 255), alpha, torch.zeros_like(alpha))
                logt = torch.cumsum(torch.log1p(-alpha), 1)
                if take >= len(own) or bool((logt[:, -1] < math.log(1e-4)).all()):
                    break
                take *= 4
            live = logt >= math.log(1e-4)
            a = torch.where(live, alpha, torch.zeros_like(alpha))
            lt = torch.cumsum(torch.log1p(-a), 1)
            last = torch.exp(lt[:, -1]) if c.shape[0] else torch.ones_like(px[:, 0])
            before = torch.exp(torch.cat([torch.zeros_like(px), lt[:, :-1]], 1)) if c.shape[0] else lt
            out = (a * before) @ c[:, 6:9] + last[:, None] * bg
            tile = out.detach().T.reshape(3, y1 - y0, x1 - x0)
            image[:, y0:y1, x0:x1] = tile
            T[y0:y1, x0:x1] = last.detach().reshape(y1 - y0, x1 - x0)
            if upstream and c.shape[0]:
                dl = upstream(tile, slice(y0, y1), slice(x0, x1)).reshape(3, -1).T
                grad[:, :9].index_add_(0, order[own[:take]], torch.autograd.grad((out * dl).sum(), c)[0])
    return image, T, grad


def _attributes64(splats):
    return [t.double() for t in (splats.means, splats.scales, splats.quats, splats.opacities, splats.sh)]


def _chain64(splats, cam, kernel, keep, grad2d):
    """Gradients w.r.t. the activated attributes from the gradients w.r.t. the projected ones."""
    idx = keep.nonzero()[:, 0]
    full = _attributes64(splats)
    sub = [t[idx].requires_grad_(True) for t in full]
    p = _project64(sub[0], sub[1], sub[2], sub[4], cam, kernel)
    g = grad2d[idx].double()
    loss = (p.u * g[:, :2]).sum() + (p.conic * g[:, 2:5]).sum() + (sub[3] * g[:, 5]).sum() + (p.rgb * g[:, 6:9]).sum()
    out = [torch.zeros_like(t) for t in full]
    for o, d in zip(out, torch.autograd.grad(loss, sub)):
        o[idx] = d
    return out


def _adam64(params, state, grads, sh):
    """One Adam step on the raw parameters from gradients w.r.t. the activated ones."""
    f32 = lambda v: float(np.float32(v))  # noqa: E731  the calls take 32-bit rates
    s, o = params.scales.double(), params.opacities.double()
    raw = dict(means=grads[0], scales=grads[1] * s, quats=grads[2], opac=grads[3] * o * (1 - o), sh=grads[4])
    names = dict(means="means", scales="log_scales", quats="quats", opac="opacity_logits", sh="sh")
    rate = torch.full((sh.shape[1], 1), f32(LRS[5]), dtype=torch.float64, device=DEV)
    rate[0] = f32(LRS[4])
    rates = dict(means=f32(LRS[0]), scales=f32(LRS[1]), quats=f32(LRS[2]), opac=f32(LRS[3]), sh=rate)
    b1, b2, out = f32(BETA1), f32(BETA2), {}
    for f, g in raw.items():
        m = b1 * getattr(state, "m_" + f).double() + (1 - b1) * g
        v = b2 * getattr(state, "v_" + f).double() + (1 - b2) * g * g
        step = (m / (1 - b1 ** STEP)) / (torch.sqrt(v / (1 - b2 ** STEP)) + f32(EPS))
        out[names[f]] = getattr(params, names[f]).double() - rates[f] * step
        out["m_" + f], out["v_" + f] = m, v
    out["scales"], out["opacities"] = torch.exp(out["log_scales"]), torch.sigmoid(out["opacity_logits"])
    return out


def _blur64(t):
    k = torch.exp(-(torch.arange(-5, 6, dtype=torch.float64, device=DEV) ** 2) / 4.5)
    k = k / k.sum()
    p = torch.nn.functional.pad(t, (5, 5, 5, 5))
    r = sum(k[i] * p[..., i:i + t.shape[-1]] for i in range(11))
    return sum(k[i] * r[:, i:i + t.shape[-2], :] for i in range(11))


def _density64(s):
    """Decisions in 32 bits, as they are defined; the new values in 64."""
    w, h, c = s.case["width"], s.case["height"], DENSIFY
    vis = s.radius > 0
    gx, gy = s.grad2d[:, 0] * np.float32(0.5 * w), s.grad2d[:, 1] * np.float32(0.5 * h)
    accum = torch.where(vis, s.accum + torch.sqrt(gx * gx + gy * gy), s.accum)
    count = torch.where(vis, s.count + 1, s.count)
    maxr = torch.where(vis, torch.maximum(s.max_radius, s.radius), s.max_radius)
    f = {k: torch.tensor(v, dtype=torch.float32, device=DEV) for k, v in c.items()}
    p, n = s.params, s.splats.n
    avg = torch.where(count > 0, accum / count.clamp(min=1), torch.zeros_like(accum))
    big = p.scales.max(1).values
    grow = avg >= f["grad_threshold"]
    split = grow & (big > f["dense_scale"])
    solid = p.opacities >= f["min_opacity"]
    fits = big <= f["max_world_scale"]
    child = (p.scales / f["split_scale_div"]).max(1).values <= f["max_world_scale"]
    i0 = (~split & solid & fits & (maxr.float() <= f["max_screen_radius"])).nonzero()[:, 0]
    i1 = (grow & ~split & solid & fits).nonzero()[:, 0]
    i2 = (split & solid & child).nonzero()[:, 0]
    rows = torch.cat([i0, i1, i2.repeat_interleave(2)])
    at = len(i0) + len(i1)
    out = {}
    for name in PARAMS:
        v = getattr(p, name)
        o = torch.zeros((2 * n,) + tuple(v.shape[1:]), dtype=torch.float64, device=DEV)
        o[:len(rows)] = v[rows].double()
        out[name] = o
    for name in MOMENTS:
        v = getattr(s.state, name)
        o = torch.zeros((2 * n,) + tuple(v.shape[1:]), dtype=torch.float64, device=DEV)
        o[:len(i0)] = v[i0].double()
        out[name] = o
    two = i2.repeat_interleave(2)
    q = p.quats[two].double()
    q = q / q.norm(dim=1, keepdim=True)
    z = s.normals[i2].double().reshape(-1, 3) * p.scales[two].double()
    qv = q[:, 1:]
    turned = z + 2 * torch.linalg.cross(qv, torch.linalg.cross(qv, z, dim=1) + q[:, :1] * z, dim=1)
    out["means"][at:len(rows)] += turned
    out["log_scales"][at:len(rows)] -= math.log(c["split_scale_div"])
    out["scales"][at:len(rows)] = torch.exp(out["log_scales"][at:len(rows)])
    return dict(n_out=None, accum=accum.double(), count=count.double(), max_radius=None, **out)


def exact(case, seed):
    op = case["op"]
    if op == "sort":
        return None  # whole numbers only
    if op == "batch":
        splats, _ = _scene(case, seed)
        att, images = _attributes64(splats), []
        for cam in _cameras(case, seed):
            p = _project64(att[0], att[1], att[2], att[4], cam, case["kernel"])
            images.append(_composite64(p, att[3], cam, case["kernel"], _visible64(p, cam, case["tile"], case["kernel"]))[0])
        return dict(images=images, num=None, status=None)
    if op in ("dssim", "density", "chain_adam", "train", "autograd", "composite_bwd"):
        s = prepare(case, seed)
        if op == "dssim":
            x, y = s.image.double().requires_grad_(True), s.target.double()
            mx, my = _blur64(x), _blur64(y)
            c1, c2 = float(np.float32(0.01) * np.float32(0.01)), float(np.float32(0.03) * np.float32(0.03))
            sxx, syy, sxy = _blur64(x * x) - mx * mx, _blur64(y * y) - my * my, _blur64(x * y) - mx * my
            ssim = (((2 * mx * my + c1) * (2 * sxy + c2)) / ((mx * mx + my * my + c1) * (sxx + syy + c2))).mean()
            lam = float(np.float32(LAMBDA))
            loss = (1 - lam) * (x - y).abs().mean() + lam * (1 - ssim)
            return dict(grad=torch.autograd.grad(loss, x)[0], loss=torch.stack([loss.detach(), ssim.detach()]))
        if op == "density":
            return _density64(s)
        if op == "chain_adam":
            g = _chain64(s.splats, s.cam, case["kernel"], _inside(s.splats, s.cam), s.grad2d)
            return dict(zip(("dmeans", "dscales", "dquats", "dopacities", "dsh"), g),
                        **_adam64(s.params, s.state, g, s.splats.sh))
        splats, cam = s.splats, s.cam
    else:
        splats, _ = _scene(case, seed)
        cam = _camera(case, seed)
    kernel = case["kernel"]
    att = _attributes64(splats)
    p = _project64(att[0], att[1], att[2], att[4], cam, kernel)
    keep = _visible64(p, cam, case["tile"], kernel)
    if op == "project":
        def kept(t):
            return torch.where(keep.view(-1, *[1] * (t.dim() - 1)), t, torch.zeros_like(t))
        return dict(depth=kept(p.depth), mean2d=kept(p.u), conic_o=kept(torch.cat([p.conic, att[3][:, None]], 1)),
                    rgb=kept(p.rgb), radius=None, tile_rect=None, tiles_touched=None, tile_runs=None, clamped=None)
    if op in ("forward", "composite"):
        image, T, _ = _composite64(p, att[3], cam, kernel, keep)
        out = dict(image=image, t_final=T, last=None, n_contrib=None)
        return dict(out, ranges=None, num=None, radius=None) if op == "forward" else out
    if op == "train":
        target, scale = s.target.double(), 1.0 / (3 * cam.width * cam.height)

        def upstream(tile, ys, xs):
            return torch.sign(tile - target[:, ys, xs]) * scale
        image, _, grad = _composite64(p, att[3], cam, kernel, keep, upstream)
        loss = (image - target).abs().mean().reshape(1)
        g = _chain64(splats, cam, kernel, keep, grad)
        return dict(loss=loss, **_adam64(s.params, s.state, g, splats.sh))
    dl = s.dl.double()
    image, _, grad = _composite64(p, att[3], cam, kernel, keep, lambda tile, ys, xs: dl[:, ys, xs])
    if op == "composite_bwd":
        return dict(grad2d=grad)
    g = _chain64(splats, cam, kernel, keep, grad)
    return dict(image=image, **dict(zip(("means", "scales", "quats", "opacities", "sh"), g)))
