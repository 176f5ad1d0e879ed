"""The render kernels over 8x8 pixel blocks, at the places where they can go
wrong: every tile shape made of such blocks, images that cut blocks, both
channel counts, square and tight lists, opacities past the clamp, conics next
to singular, colours that are not finite.  Images within 1e-5 and gradients
within 1e-4 relative L2 of the FP64 oracle, as in test_gpu_parity.py."""
import numpy as np
import pytest
import torch

import oracle
from paper_2409_13055_gb300 import binding as B
from paper_2409_13055_gb300 import mapping, scenes
from tests import gpu_util as U

pytestmark = pytest.mark.gpu

IMG_TOL, GRAD_TOL = 1e-5, 1e-4
BG = (0.1, 0.2, 0.3)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_13055_gb300 import build
    build.build()
    B.lib()


def _check(p, view, tile, **kw):
    target = scenes.random_target(view, 17)
    proj, st, lst, o = oracle.forward_view(p, view, tile[0], tile[1], BG)
    gm = mapping.GaussianMap(p)
    rast = mapping.Rasterizer([view], gm.n, instance_capacity=1 << 20, tile=tile, bg=BG, **kw)
    rast.forward(gm.gs_map())
    torch.cuda.synchronize()
    assert rast.counters().status == 0
    ok = ~U.guard_pixel_mask(view, proj, o, tile)
    assert ok.mean() > 0.8
    img = rast.view_slice(rast.images, 0).cpu().numpy()
    assert np.abs(img - o["image"])[:, ok].max() <= IMG_TOL
    T = rast.view_slice(rast.final_T, 0, per_pixel=True).cpu().numpy()
    assert np.abs(T - o["final_T"])[ok].max() <= IMG_TOL
    _, dimg = oracle.loss_l1_ssim(o["image"], target, 0.2)
    dimg = dimg * (ok & ~U.grad_pixel_mask(o))[None]
    og = oracle.project_bwd(p, view, oracle.render_bwd(proj, st, lst, view, dimg, tile[0], tile[1],
                                                       BG), tile_w=tile[0], tile_h=tile[1])
    rast.render_bwd(gm.gs_map(), gm.gs_map_grad(), dL=rast.pack([dimg]))
    torch.cuda.synchronize()
    kink = (proj["guard"] & oracle.GUARD_KINK) != 0
    errs = U.grad_errors({k: v.cpu().numpy() for k, v in gm.grads().items()}, og, ~kink)
    assert all(e <= GRAD_TOL for e in errs.values()), errs


@pytest.mark.parametrize("channels", [3, 1])
@pytest.mark.parametrize("tile", [(8, 8), (16, 8), (8, 16), (16, 16), (32, 8), (8, 32)])
def test_every_tile_of_blocks_at_ragged_sizes(tile, channels):
    p, view = scenes.tiny_scene(900, 97, 61, seed=71, sh_degree=1)
    view = dict(view, channels=channels)
    _check(p, view, tile)
    _check(p, view, tile, tight_rect=False)


@pytest.mark.parametrize("size", [(1, 1), (7, 9), (9, 8), (17, 3)])
def test_images_smaller_than_a_few_blocks(size):
    p, view = scenes.tiny_scene(120, size[0], size[1], seed=72, log_scale=(-2.5, 0.3))
    _check(p, view, (8, 8))
    _check(p, view, (16, 16))


@pytest.mark.parametrize("tile", [(8, 8), (16, 16)])
def test_opacities_past_the_clamp(tile):
    p, view = scenes.tiny_scene(400, 96, 64, seed=73)
    p["opacity_logits"] = np.random.default_rng(5).uniform(-2.0, 9.0, 400).astype(np.float32)
    _check(p, view, tile)


def test_needles_render_as_the_tile_kernels_render_them():
    """Conics next to singular, where rounding can make a power positive, among
    ordinary Gaussians and alone, opaque ones among them: a deterministic plan
    of 16x16 tiles renders with the kernels of gs_render.cu, whose decisions
    and rounding the block kernels repeat bit for bit."""
    p, view = scenes.tiny_scene(400, 96, 64, seed=73)
    p["opacity_logits"] = np.random.default_rng(5).uniform(-2.0, 9.0, 400).astype(np.float32)
    p["log_scales"][::5] = np.array([-8.0, -1.0, -8.0], np.float32)
    p["log_scales"][1::25] = np.array([-8.0, 4.0, -8.0], np.float32)
    for q in (p, scenes.subset(p, np.arange(0, 400, 5)), scenes.subset(p, np.arange(1, 400, 25))):
        gm = mapping.GaussianMap(q)
        out = []
        for kw in (dict(), dict(deterministic=True, pixels_per_thread_bwd=8)):
            rast = mapping.Rasterizer([view], gm.n, instance_capacity=1 << 20, bg=BG, **kw)
            rast.forward(gm.gs_map())
            out.append([t.cpu().numpy() for t in (rast.images, rast.final_T, rast.last_idx)])
        for x, y in zip(*out):
            np.testing.assert_array_equal(x, y)


def test_a_colour_that_is_not_finite_stays_in_its_blocks():
    p, view = scenes.tiny_scene(300, 64, 64, seed=74, depth=(2.0, 3.0))
    proj = oracle.project(p, view, 8, 8)
    g = int(np.argmin(np.hypot(*(proj["mean2d"] - np.array([12.0, 12.0])).T)
                      + 1e9 * (proj["tiles_touched"] == 0)))
    p["sh"][0, g] = np.inf
    gm = mapping.GaussianMap(p)
    rast = mapping.Rasterizer([view], gm.n, instance_capacity=1 << 18, tile=(8, 8))
    rast.forward(gm.gs_map())
    img = rast.view_slice(rast.images, 0).cpu().numpy()
    reach = int(proj["radius"][g]) + 8
    cx, cy = proj["mean2d"][g]
    yy, xx = np.mgrid[0:64, 0:64]
    far = (np.abs(xx - cx) > reach) | (np.abs(yy - cy) > reach)
    assert far.mean() > 0.3 and np.isfinite(img[:, far]).all()
