"""What a user of this framework has it do, as cases that can be timed and compared.

A mapping program holds a Gaussian map, cameras and target images.  It plans a
rasteriser once per set of views, captures its mapping iteration as a CUDA
graph and replays it; it renders views without optimising; it differentiates
through the PyTorch autograd functions; and for each new keyframe it picks
pixels, triangulates them and builds the target's pyramid.  The listed cases
cover these calls from the smallest workload of the repository (10k Gaussians,
320x240) to its largest (2M Gaussians under a window of eight keyframes), at
the launch shape a rasteriser has by default (16x16 tiles) and at the one the
autotuner picks on this GPU (8x8 tiles), in colour and in gray, at SH degrees
0 to 3, with and without the density statistic and checkpointing.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2409_13055_gb300 import mapping, pointcloud, pyramid, scenes

# the autotuner's launch shape on this GPU (8x8 tiles, forward and backward apart)
TUNED = dict(tile=(8, 8), smem_batch=128, pixels_per_thread=1, smem_batch_bwd=64,
             pixels_per_thread_bwd=2)
# the learning rates late in a run: the map stays what it was while it is timed
LATE = {k: 0.01 * v for k, v in mapping.DEFAULT_LR.items()}
BETA1, BETA2, EPS = 0.9, 0.999, 1e-15
DEV = "cuda"


def listed():
    return [
        # a preview render of the smallest map, launched call by call
        dict(name="forward_10k_320x240", kind="forward", scene="planes", n=10_000, degree=0,
             width=320, height=240, focal=300.0, channels=3, views="one", tuned=False),
        # the smallest mapping iteration, L1 loss: launches and latency count
        dict(name="step_10k_320x240", kind="step", scene="planes", n=10_000, degree=0, width=320,
             height=240, focal=300.0, channels=3, views="one", tuned=False, lam=0.0,
             recompute=0, stats=False),
        # an ordinary indoor keyframe at the default launch shape
        dict(name="step_200k_640x480", kind="step", scene="room", n=200_000, degree=3, width=640,
             height=480, focal=525.0, channels=3, views="one", tuned=False, lam=0.2,
             recompute=0, stats=False),
        # the same map differentiated through PyTorch, at the autotuned launch shape
        dict(name="autograd_200k_640x480", kind="autograd", scene="room", n=200_000, degree=3,
             width=640, height=480, focal=525.0, channels=3, views="one", tuned=True, lam=0.2),
        # a render of a map of ragged size for display, gray, default launch shape
        dict(name="forward_70k_751x479_gray", kind="forward", scene="room", n=70_001, degree=1,
             width=751, height=479, focal=460.0, channels=1, views="one", tuned=False),
        # the densification phase: iterations that also gather the density statistic
        dict(name="step_stats_350k_1037x563", kind="step", scene="room", n=350_003, degree=2,
             width=1037, height=563, focal=560.0, channels=3, views="one", tuned=False, lam=0.2,
             recompute=0, stats=True),
        # the headline: one million Gaussians, one 1200x680 view
        dict(name="step_1M_1200x680", kind="step", scene="room", n=1_000_000, degree=3,
             width=1200, height=680, focal=600.0, channels=3, views="one", tuned=True, lam=0.2,
             recompute=0, stats=False),
        # sixteen keyframes of mixed resolution in one batch
        dict(name="step_500k_16views", kind="step", scene="room", n=500_000, degree=3, width=0,
             height=0, focal=0.0, channels=0, views="mixed16", tuned=True, lam=0.2, recompute=0,
             stats=False),
        # streaming: a window of eight gray keyframes over the grown map, checkpointed
        dict(name="step_2M_window8", kind="step", scene="stream", n=2_000_000, degree=3,
             width=752, height=480, focal=460.0, channels=1, views="window8", tuned=True,
             lam=0.2, recompute=4, stats=False),
        # the photometric loss and its gradient for a user's own rendered image
        dict(name="loss_1200x680", kind="loss", width=1200, height=680, channels=3, lam=0.2),
        # one optimiser step of a running map
        dict(name="adam_600k", kind="adam", n=600_000, degree=3, visible=1.0),
        # a keyframe arrives: target pyramid, tracked pixels, triangles, new Gaussians
        dict(name="keyframe_752x480", kind="keyframe", width=752, height=480, focal=460.0,
             levels=3, block=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case of the ranges above."""
    kind = rng.choice(["forward", "forward", "step", "step", "step", "autograd", "loss", "adam",
                       "keyframe"])
    if kind == "adam":
        return dict(kind=kind, n=_log(rng, 10_000, 1_500_000), degree=rng.randint(0, 3),
                    visible=rng.choice([1.0, round(rng.uniform(0.2, 0.8), 2)]))
    px = math.exp(rng.uniform(math.log(320 * 240), math.log(1200 * 680)))
    aspect = rng.uniform(1.2, 1.8)
    width, height = int(round(math.sqrt(px * aspect))), int(round(math.sqrt(px / aspect)))
    if kind == "loss":
        return dict(kind=kind, width=width, height=height, channels=rng.choice([1, 3]),
                    lam=round(rng.uniform(0.0, 0.4), 2))
    if kind == "keyframe":
        return dict(kind=kind, width=width, height=height, focal=round(0.6 * width, 1),
                    levels=rng.randint(2, 4), block=rng.choice([4, 5, 6]))
    tuned = rng.random() < 0.5
    case = dict(kind=kind, scene="room", n=_log(rng, 10_000, 1_000_000), degree=rng.randint(0, 3),
                width=width, height=height, focal=round(rng.uniform(0.5, 0.9) * width, 1),
                channels=rng.choice([1, 3, 3]), views="one", tuned=tuned)
    if kind == "forward":
        return case
    case["lam"] = rng.choice([0.0, 0.2, 0.2])
    if kind == "autograd":
        return case
    case.update(recompute=0, stats=rng.random() < 0.25)
    if rng.random() < 0.4:
        case.update(views="several", width=min(width, 800), height=min(height, 600),
                    n=min(case["n"], 400_000), recompute=rng.choice([0, 2]))
    return case


# --------------------------------------------------------------------------
# Inputs, from the seed alone.
# --------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _room_points(n, seed, g):
    """n points sampled area-uniformly on a box room and 20 boxes on its floor."""
    rng = np.random.default_rng(seed)
    faces = []

    def box(lo, hi):
        d = np.asarray(hi, float) - lo
        ex, ey, ez = np.diag(d)
        faces.extend([(lo, ex, ey), (lo + ez, ex, ey), (lo, ey, ez), (lo + ex, ey, ez),
                      (lo, ex, ez), (lo + ey, ex, ez)])

    box(np.array([-3.0, -1.5, -1.0]), np.array([3.0, 1.5, 5.0]))
    for _ in range(20):
        s = rng.uniform(0.2, 1.0, 3)
        lo = np.array([rng.uniform(-2.4, 2.4) - s[0] / 2, 1.5 - s[1],
                       rng.uniform(1.2, 4.4) - s[2] / 2])
        box(lo, lo + s)
    area = np.array([np.linalg.norm(np.cross(u, v)) for (_, u, v) in faces])
    f = torch.multinomial(torch.tensor(area, device=DEV), n, replacement=True, generator=g)
    O, U, V = (torch.tensor(np.stack([x[k] for x in faces]), device=DEV, dtype=torch.float32)
               for k in range(3))
    return O[f] + _rand(g, n, 1) * U[f] + _rand(g, n, 1) * V[f]


def _map_tensors(case, seed):
    """The map of a case as float32 tensors on the GPU."""
    g, n, K = _gen(seed), case["n"], (case["degree"] + 1) ** 2
    quats = _randn(g, n, 4)
    logits = _randn(g, n)
    if case["scene"] == "planes":
        # pixels back-projected onto three planes, not turned, flat colours (of
        # unequal scales, as they are after the first iterations: a sphere's
        # rotation has no gradient but rounding errors)
        iz = torch.tensor([[0.45, 0.05, -0.04], [0.55, -0.06, 0.08], [0.65, 0.03, 0.02]],
                          device=DEV)[torch.randint(0, 3, (n,), generator=g, device=DEV)]
        xn = (_rand(g, n) - 0.5) * case["width"] / case["focal"]
        yn = (_rand(g, n) - 0.5) * case["height"] / case["focal"]
        z = (1.0 / (iz[:, 0] + iz[:, 1] * xn + iz[:, 2] * yn)).clamp(1.0, 4.0)
        means = torch.stack([xn * z, yn * z, z], 1)
        ls = -4.0 + 0.3 * _randn(g, n, 3)
        quats = torch.tensor([1.0, 0.0, 0.0, 0.0], device=DEV).expand(n, 4)
        sh = torch.zeros(K, n, 3, device=DEV)
        sh[0] = (2 * _rand(g, n, 3) - 1) * math.sqrt(math.pi)
    else:
        means = _room_points(n, seed, g)
        if case["scene"] == "stream":
            # in order of insertion: keyframe after keyframe round the loop, no
            # order within a keyframe; points of low opacity one block wide, a
            # little stretched by the iterations so far
            ang = torch.atan2(means[:, 2] - 1.6, means[:, 0])
            means = means[torch.argsort(ang + 0.06 * _rand(g, n))]
            ls = -5.0 + 0.3 * _randn(g, n, 1) + 0.15 * _randn(g, n, 3)
            logits = -2.0 + 0.5 * logits
        else:
            # stored along a Z-order curve, as maps that are kept are
            means = means[mapping.morton_order(means.double())]
            ls = -4.5 + 0.5 * _randn(g, n, 3)
        sh = 0.1 * _randn(g, K, n, 3)
    return dict(means=means, log_scales=ls, quats=quats, opacity_logits=logits, sh=sh,
                sh_degree=case["degree"])


def _map(case, seed):
    t = _map_tensors(case, seed)
    return mapping.GaussianMap({k: (v.contiguous().cpu().numpy() if k != "sh_degree" else v)
                                for k, v in t.items()})


def _views(case):
    if case["views"] == "mixed16":
        return scenes.views_mixed16()
    if case["views"] == "window8":
        return scenes.drone_loop(100, width=case["width"], height=case["height"],
                                 f=case["focal"])[20:28]
    w, h, f, c = case["width"], case["height"], case["focal"], case["channels"]
    if case["views"] == "several":
        rng = np.random.default_rng(7)
        out = []
        for _ in range(3):
            R, t = scenes.random_pose(rng, 0.5, 20.0)
            out.append(scenes.camera(w, h, f, f, R=R, t=t, channels=c))
        return out
    return [scenes.camera(w, h, f, f, channels=c)]


def _picture(c, h, w, seed):
    """A textured image in [0, 1]: patches of plaid of different contrast, some noise."""
    g = _gen(seed)
    y = torch.arange(h, device=DEV).view(1, h, 1) / 40.0
    x = torch.arange(w, device=DEV).view(1, 1, w) / 40.0
    k = _rand(g, 8)
    img = 0.5 + 0.2 * torch.sin(6.0 * (0.5 + k[0]) * x + 3 * k[1]) * torch.sin(
        5.0 * (0.5 + k[2]) * y + 3 * k[3])
    patch = _rand(g, c, h // 60 + 1, w // 60 + 1)
    img = img + 0.5 * (torch.nn.functional.interpolate(patch[None], size=(h, w), mode="nearest")[0]
                       - 0.5)
    return (img + 0.004 * _randn(g, c, h, w)).clamp(0, 1).contiguous()


def _targets(views, seed):
    return torch.cat([_picture(v["channels"], v["height"], v["width"], seed * 64 + i).reshape(-1)
                      for i, v in enumerate(views)])


def _rasterizer(case, views, gmap, **kw):
    if case["tuned"]:
        kw.update(TUNED)
    return mapping.fit_instance_capacity(views, gmap, headroom=1.5, **kw)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "loss":
        view = scenes.camera(case["width"], case["height"], 1.0, 1.0, channels=case["channels"])
        rast = mapping.Rasterizer([view], 1, instance_capacity=1)
        targets = _targets([view], seed)
        images = targets + 0.05 * _randn(_gen(seed + 1), targets.numel())
        return dict(kind=kind, rast=rast, targets=targets, images=images, lam=case["lam"])
    if kind == "adam":
        gmap = _map(dict(case, scene="room"), seed)
        g = _gen(seed + 1)
        gmap.grad.copy_(1e-4 * torch.randn(gmap.total, generator=g, device=DEV))
        gmap.m.copy_(1e-4 * torch.randn(gmap.total, generator=g, device=DEV))
        gmap.v.copy_(1e-8 * torch.rand(gmap.total, generator=g, device=DEV))
        gmap.step.fill_(1000)
        vis = None
        if case["visible"] < 1.0:  # runs of Gaussians in or out of view
            run = _rand(g, gmap.n // 500 + 1).repeat_interleave(500)[:gmap.n]
            vis = (run < case["visible"]).to(torch.uint8)
        return dict(kind=kind, gmap=gmap, visible=vis)
    if kind == "keyframe":
        h, w, f = case["height"], case["width"], case["focal"]
        depth = 2.0 + torch.nn.functional.interpolate(_rand(_gen(seed + 1), 1, 1, 6, 8), (h, w),
                                                      mode="bilinear")[0, 0]
        # room for the new points, and for their Gaussians on their way into the map
        most = (w // 4 + 1) * (h // 4 + 1) * 2
        slots = dict(px=torch.zeros(most, dtype=torch.int64, device=DEV),
                     py=torch.zeros(most, dtype=torch.int64, device=DEV),
                     z=torch.zeros(most, device=DEV))
        host = dict(means=np.zeros((most, 3), np.float32),
                    log_scales=np.zeros((most, 3), np.float32),
                    opacity_logits=np.zeros(most, np.float32),
                    sh=np.zeros((4, most, 3), np.float32))
        return dict(kind=kind, image=_picture(1, h, w, seed), depth=depth, levels=case["levels"],
                    block=case["block"], view=scenes.camera(w, h, f, f, channels=1), slots=slots,
                    host=host)
    views = _views(case)
    if kind == "autograd":
        t = _map_tensors(case, seed)
        leaves = [t[k].contiguous().requires_grad_() for k in
                  ("means", "log_scales", "quats", "opacity_logits", "sh")]
        rast = _rasterizer(case, views, _map(case, seed))
        return dict(kind=kind, leaves=leaves, rast=rast, targets=_targets(views, seed),
                    lam=case["lam"])
    gmap = _map(case, seed)
    if kind == "forward":
        return dict(kind=kind, rast=_rasterizer(case, views, gmap), gmap=gmap)
    rast = _rasterizer(case, views, gmap, recompute=case["recompute"], density_stats=case["stats"])
    stats = None
    if case["stats"]:
        stats = tuple(torch.zeros(gmap.n, device=DEV) for _ in range(2))
    step = mapping.MappingStep(gmap, rast, _targets(views, seed), case["lam"], lr=LATE,
                               stats=stats)
    start = gmap.data.clone()
    step.capture()
    # the warm-up iterations of the capture are taken back: the first pass is
    # the map's first iteration
    gmap.data.copy_(start)
    for buf in (gmap.m, gmap.v, gmap.step) + (stats or ()):
        buf.zero_()
    return dict(kind=kind, step=step, gmap=gmap, rast=rast, stats=stats)


def _by_group(gmap, buf):
    n, o, K = gmap.n, gmap.off, gmap.K
    return dict(means=buf[o["means"]:o["means"] + 3 * n],
                log_scales=buf[o["log_scales"]:o["log_scales"] + 3 * n],
                quats=buf[o["quats"]:o["quats"] + 4 * n],
                opacity_logits=buf[o["opacity_logits"]:o["opacity_logits"] + n],
                sh=buf[o["sh"]:o["sh"] + 3 * K * n])


def run(state):
    kind = state["kind"]
    if kind == "step":
        state["step"]()
        gmap, rast = state["gmap"], state["rast"]
        out = dict(images=rast.images, loss=rast.loss, params=_by_group(gmap, gmap.data),
                   m=_by_group(gmap, gmap.m), v=_by_group(gmap, gmap.v))
        if state["stats"]:
            out["stats"] = list(state["stats"])
        return out
    if kind == "forward":
        rast = state["rast"]
        rast.forward(state["gmap"].gs_map())
        return dict(images=rast.images, final_T=rast.final_T, last_idx=rast.last_idx)
    if kind == "autograd":
        for t in state["leaves"]:
            t.grad = None
        images = mapping.GSRender.apply(*state["leaves"], state["rast"])
        loss = mapping.L1SSIMLoss.apply(images, state["targets"], state["rast"], state["lam"])
        loss.backward()
        return dict(images=images, loss=loss, grads=[t.grad for t in state["leaves"]])
    if kind == "loss":
        rast = state["rast"]
        rast.loss_l1_ssim(state["targets"], state["lam"], images=state["images"])
        return dict(loss=rast.loss, dL=rast.dL)
    if kind == "adam":
        gmap = state["gmap"]
        gmap.adam_step(visible=state["visible"])
        return dict(params=_by_group(gmap, gmap.data), m=_by_group(gmap, gmap.m),
                    v=_by_group(gmap, gmap.v))
    image, depth, slots, host = (state[k] for k in ("image", "depth", "slots", "host"))
    levels = pyramid.pyramid(image, state["levels"])
    points = pointcloud.keyframe_points(image[0], lambda x, y: depth[y, x], block=state["block"])
    new = pointcloud.gaussians_from_points(state["view"], *points, image[0], sh_degree=1)
    k = points[0].numel()
    for slot, value in zip(slots.values(), points):
        slot[:k] = value
    for name, slot in host.items():
        if name == "sh":
            slot[:, :k] = new[name]
        else:
            slot[:k] = new[name]
    return dict(levels=levels[1:], count=k, points=slots, new=host)


def work(case):
    """Bytes and operations of one pass: inputs read once, outputs written once;
    a (pixel, Gaussian) pair costs about 20 operations to blend and 60 more to
    differentiate."""
    kind = case["kind"]
    if kind == "loss":
        v = case["width"] * case["height"] * case["channels"]
        return dict(bytes=12.0 * v, flops=400.0 * v)
    if kind == "keyframe":
        v = case["width"] * case["height"]
        return dict(bytes=16.0 * v, flops=100.0 * v)
    floats = case["n"] * (11 + 3 * (case["degree"] + 1) ** 2)
    if kind == "adam":
        return dict(bytes=28.0 * floats * case["visible"], flops=15.0 * floats)
    views = _views(case)
    values = sum(v["width"] * v["height"] * v["channels"] for v in views)
    pixels = sum(v["width"] * v["height"] for v in views)
    # the visible half of the map, some 60 pixels each that blend it, at most
    # what a pixel takes before it is opaque
    pairs = sum(min(30.0 * case["n"], 60.0 * v["width"] * v["height"]) for v in views)
    if kind == "forward":
        return dict(bytes=4.0 * (floats + values + 2 * pixels), flops=20.0 * pairs)
    if kind == "autograd":
        return dict(bytes=4.0 * (2 * floats + 2 * values), flops=80.0 * pairs)
    return dict(bytes=4.0 * (6 * floats + 2 * values), flops=80.0 * pairs)


# --------------------------------------------------------------------------
# The same results in 64 bits, in plain torch.
# --------------------------------------------------------------------------
def _sh_basis(d, degree):
    x, y, z = d.unbind(1)
    Y = [torch.full_like(x, 0.28209479177387814)]
    if degree >= 1:
        c = 0.4886025119029199
        Y += [-c * y, c * z, -c * x]
    if degree >= 2:
        a, b, c = 1.0925484305920792, 0.31539156525252005, 0.5462742152960396
        Y += [a * x * y, -a * y * z, b * (2 * z * z - x * x - y * y), -a * x * z,
              c * (x * x - y * y)]
    if degree >= 3:
        a, b, c, d3, e = (0.5900435899266435, 2.890611442640554, 0.4570457994644658,
                          0.3731763325901154, 1.445305721320277)
        q = 4 * z * z - x * x - y * y
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * q,
              d3 * z * (2 * z * z - 3 * x * x - 3 * y * y), -c * x * q, e * z * (x * x - y * y),
              -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _project64(P, degree, view, tile):
    """Projected Gaussians of one view (differentiable), their tile rects, depth order."""
    means, ls, quats, logits, sh = P
    R = torch.tensor(np.asarray(view["R"], np.float64), device=DEV)
    t = torch.tensor(np.asarray(view["t"], np.float64), device=DEV)
    fx, fy, cx, cy = (float(np.float32(view[k])) for k in ("fx", "fy", "cx", "cy"))
    W, H = view["width"], view["height"]
    xc = means @ R.T + t
    keep = (xc[:, 2].float() > float(np.float32(0.2))).nonzero()[:, 0]
    xc, means, ls, quats, logits, sh = (xc[keep], means[keep], ls[keep], quats[keep],
                                        logits[keep], sh[:, keep])
    x, y, z = xc.unbind(1)
    mu = torch.stack([fx * x / z + cx, fy * y / z + cy], 1)
    u = (x / z).clamp(-1.3 * cx / fx, 1.3 * (W - cx) / fx)
    v = (y / z).clamp(-1.3 * cy / fy, 1.3 * (H - cy) / fy)
    T0 = (fx / z)[:, None] * R[0] - (fx * u / z)[:, None] * R[2]
    T1 = (fy / z)[:, None] * R[1] - (fy * v / z)[:, None] * R[2]
    q = quats / quats.norm(dim=1, keepdim=True)
    w, i, j, k = q.unbind(1)
    Rq = torch.stack([1 - 2 * (j * j + k * k), 2 * (i * j - w * k), 2 * (i * k + w * j),
                      2 * (i * j + w * k), 1 - 2 * (i * i + k * k), 2 * (j * k - w * i),
                      2 * (i * k - w * j), 2 * (j * k + w * i), 1 - 2 * (i * i + j * j)],
                     1).view(-1, 3, 3)
    M = Rq * ls.exp()[:, None, :]
    A0, A1 = (T0[:, None, :] @ M)[:, 0], (T1[:, None, :] @ M)[:, 0]
    a, b, c = (A0 * A0).sum(1) + 0.3, (A0 * A1).sum(1), (A1 * A1).sum(1) + 0.3
    det = a * c - b * b
    centre = -(R.T @ t)
    d = means - centre
    d = d / d.norm(dim=1, keepdim=True)
    col = ((_sh_basis(d, degree).T[:, :, None] * sh).sum(0) + 0.5).clamp_min(0.0)
    feat = torch.cat([mu, torch.stack([c / det, -b / det, a / det, torch.sigmoid(logits)], 1),
                      col], 1)
    with torch.no_grad():
        mid = 0.5 * (a + c)
        rad = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp_min(0))))
        lo = torch.floor((mu - rad[:, None]) / torch.tensor(tile, device=DEV))
        hi = torch.floor((mu + rad[:, None] + torch.tensor(tile, device=DEV) - 1)
                         / torch.tensor(tile, device=DEV))
        # pixels [lo, hi) of whole tiles, and the box that alpha >= 1/255 stays inside
        rect = torch.cat([lo, hi], 1) * torch.tensor(tile + tile, device=DEV)
        tau = 2 * torch.log((255.0 * feat[:, 5]).clamp_min(1.0))
        ext = torch.stack([torch.sqrt(tau * a), torch.sqrt(tau * c)], 1) + 0.01
        box = torch.cat([torch.maximum(rect[:, :2], mu - ext),
                         torch.minimum(rect[:, 2:], mu + ext + 1)], 1)
        box[feat[:, 5] < 1.0 / 255] = -1.0
        order = torch.argsort(z.float(), stable=True)
    return feat[order], rect[order], box[order]


def _blend64(feat, rect, box, view, bx, by, size=32):
    """Colour and transmittance of the pixels of one block."""
    W, H = view["width"], view["height"]
    x1, y1 = min(bx + size, W), min(by + size, H)
    near = ((box[:, 0] < x1) & (box[:, 2] > bx) & (box[:, 1] < y1) & (box[:, 3] > by)).nonzero()
    f, r = feat[near[:, 0]], rect[near[:, 0]]
    py, px = torch.meshgrid(torch.arange(by, y1, device=DEV, dtype=torch.float64),
                            torch.arange(bx, x1, device=DEV, dtype=torch.float64), indexing="ij")
    px, py = px.reshape(1, -1), py.reshape(1, -1)
    dx, dy = f[:, 0:1] - px, f[:, 1:2] - py
    power = -0.5 * (f[:, 2:3] * dx * dx + f[:, 4:5] * dy * dy) - f[:, 3:4] * dx * dy
    alpha = (f[:, 5:6] * torch.exp(power)).clamp_max(0.99)
    ok = ((power <= 0) & (alpha >= 1.0 / 255) & (px >= r[:, 0:1]) & (px < r[:, 2:3])
          & (py >= r[:, 1:2]) & (py < r[:, 3:4]))
    alpha = torch.where(ok, alpha, torch.zeros_like(alpha))
    T = torch.cumprod(1 - alpha, 0)
    alpha = torch.where(T.detach() >= 1e-4, alpha, torch.zeros_like(alpha))
    T = torch.cumprod(1 - alpha, 0)
    before = torch.cat([torch.ones_like(T[:1]), T[:-1]], 0)
    col = (alpha * before).T @ f[:, 6:9]
    last = T[-1] if T.shape[0] else torch.ones_like(px[0])
    if view["channels"] == 1:
        col = col.mean(1, keepdim=True)
    return col.T.reshape(-1, y1 - by, x1 - bx), last.reshape(y1 - by, x1 - bx)


def _blocks(view, size=32):
    return [(bx, by) for by in range(0, view["height"], size)
            for bx in range(0, view["width"], size)]


def _render64(P, degree, view, tile):
    img = torch.zeros(view["channels"], view["height"], view["width"], dtype=torch.float64,
                      device=DEV)
    T = torch.ones(view["height"], view["width"], dtype=torch.float64, device=DEV)
    with torch.no_grad():
        F = _project64(P, degree, view, tile)
        for bx, by in _blocks(view):
            c, t = _blend64(*F, view, bx, by)
            img[:, by:by + t.shape[0], bx:bx + t.shape[1]] = c
            T[by:by + t.shape[0], bx:bx + t.shape[1]] = t
    return img, T


def _loss64(img, tgt, lam):
    """(1 - lam) mean|I - G| + lam (1 - mean SSIM), 11x11 window of sigma 1.5, zero padding."""
    w = torch.exp(-(torch.arange(11, device=DEV, dtype=torch.float64) - 5) ** 2 / 4.5)
    w = w / w.sum()

    def blur(x):
        x = torch.nn.functional.conv2d(x[:, None], w.view(1, 1, 1, 11), padding=(0, 5))
        return torch.nn.functional.conv2d(x, w.view(1, 1, 11, 1), padding=(5, 0))[:, 0]

    mx, my = blur(img), blur(tgt)
    vx, vy, cxy = blur(img * img) - mx * mx, blur(tgt * tgt) - my * my, blur(img * tgt) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    s = (2 * mx * my + c1) * (2 * cxy + c2) / ((mx * mx + my * my + c1) * (vx + vy + c2))
    return (1 - lam) * (img - tgt).abs().mean() + lam * (1 - s.mean())


def _gradients64(P, degree, views, targets, tile, lam):
    """Images, loss and parameter gradients of the mean loss over the views."""
    total = [torch.zeros_like(p) for p in P]
    images, loss, at = [], 0.0, 0
    for view in views:
        img, _ = _render64(P, degree, view, tile)
        tgt = targets[at:at + img.numel()].double().view(img.shape)
        at += img.numel()
        leaf = img.clone().requires_grad_()
        L = _loss64(leaf, tgt, lam) / len(views)
        L.backward()
        dimg = leaf.grad
        Q = [p.detach().clone().requires_grad_() for p in P]
        feat, rect, box = _project64(Q, degree, view, tile)
        flat = feat.detach().clone().requires_grad_()
        for bx, by in _blocks(view):
            c, t = _blend64(flat, rect, box, view, bx, by)
            if c.requires_grad:
                (c * dimg[:, by:by + t.shape[0], bx:bx + t.shape[1]]).sum().backward()
        if flat.grad is not None:
            feat.backward(flat.grad)
            for s, q in zip(total, Q):
                s += q.grad
        images.append(img.reshape(-1))
        loss += float(L)
    return torch.cat(images), loss, total


def exact(case, seed):
    kind = case["kind"]
    if kind == "keyframe":
        x = _picture(1, case["height"], case["width"], seed).double()
        w = torch.tensor([1.0, 4.0, 6.0, 4.0, 1.0], device=DEV, dtype=torch.float64) / 16
        levels = []
        for _ in range(case["levels"] - 1):
            y = torch.nn.functional.pad(x[None], (2, 2, 2, 2), mode="reflect")
            y = torch.nn.functional.conv2d(y, w.view(1, 1, 1, 5))
            x = torch.nn.functional.conv2d(y, w.view(1, 1, 5, 1))[0][:, ::2, ::2]
            levels.append(x)
        # the interpolated depths depend on which of several valid triangulations is taken
        return dict(levels=levels, count=None, points=None, new=None)
    if kind == "loss":
        s = prepare(case, seed)
        shape = (case["channels"], case["height"], case["width"])
        img = s["images"].double().view(shape).requires_grad_()
        L = _loss64(img, s["targets"].double().view(shape), case["lam"])
        L.backward()
        return dict(loss=L.detach().reshape(1), dL=img.grad.reshape(-1))
    if kind == "adam":
        s = prepare(case, seed)
        gmap = s["gmap"]
        p, g, m, v = ({k: t.double() for k, t in _by_group(gmap, b).items()}
                      for b in (gmap.data, gmap.grad, gmap.m, gmap.v))
        return _adam64(p, g, m, v, 1001, mapping.DEFAULT_LR, s["visible"], gmap.n)
    views = _views(case)
    pixels = sum(v["width"] * v["height"] for v in views)
    if case["n"] > 1_000_000 or pixels > 1_000_000:
        return None
    tile = (8.0, 8.0) if case["tuned"] else (16.0, 16.0)
    t = _map_tensors(case, seed)
    P = [t[k].double() for k in ("means", "log_scales", "quats", "opacity_logits", "sh")]
    if kind == "forward":
        img, T = _render64(P, case["degree"], views[0], tile)
        return dict(images=img.reshape(-1), final_T=T.reshape(-1), last_idx=None)
    images, loss, grads = _gradients64(P, case["degree"], views, _targets(views, seed), tile,
                                       case["lam"])
    if kind == "autograd":
        return dict(images=images, loss=loss, grads=grads)
    names = ("means", "log_scales", "quats", "opacity_logits", "sh")
    p = {k: x.reshape(-1) for k, x in zip(names, P)}
    g = {k: x.reshape(-1) for k, x in zip(names, grads)}
    zero = {k: torch.zeros_like(x) for k, x in p.items()}
    out = dict(images=images, loss=torch.tensor([loss], dtype=torch.float64),
               **_adam64(p, g, zero, zero, 1, LATE, None, case["n"]))
    # a first step moves every parameter by its rate times the gradient's sign,
    # which is no value for a gradient of rounding errors alone
    out["params"] = {k: None for k in names}
    if case["stats"]:
        out["stats"] = [None, None]
    return out


def _adam64(p, g, m, v, t, lr, visible, n):
    b1, b2 = float(np.float32(BETA1)), float(np.float32(BETA2))
    out = dict(params={}, m={}, v={})
    for k, width in (("means", 3), ("log_scales", 3), ("quats", 4), ("opacity_logits", 1),
                     ("sh", 3)):
        rate = torch.full_like(p[k], lr[k] if k != "sh" else lr["sh_rest"])
        if k == "sh":
            rate[:3 * n] = lr["sh_dc"]
        m1 = b1 * m[k] + (1 - b1) * g[k]
        v1 = b2 * v[k] + (1 - b2) * g[k] ** 2
        p1 = p[k] - rate * (m1 / (1 - b1 ** t)) / (torch.sqrt(v1 / (1 - b2 ** t)) + EPS)
        if visible is not None:
            on = visible.bool().repeat_interleave(width).repeat(p[k].numel() // (width * n))
            p1, m1, v1 = (torch.where(on, a, b) for a, b in ((p1, p[k]), (m1, m[k]), (v1, v[k])))
        out["params"][k], out["m"][k], out["v"][k] = p1, m1, v1
    return out
