"""Tiles of several blocks leave a listed Gaussian out of the blocks it cannot reach.
Long needles, whose quadratic form cancels far from the mean, must not be left
out where the pixel loop finds them: a deterministic plan of 16x16 tiles and
eight pixels per thread renders the same lists without any such test."""
import numpy as np
import pytest
import torch

from paper_2409_13055_gb300 import binding as B
from paper_2409_13055_gb300 import mapping, scenes
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_13055_gb300 import build
    build.build()
    B.lib()


def _needles(rng, n, sigma, reach, f=600.0, z=2.0):
    """n needles of about `sigma` x 0.5 pixels through the image, their means up to
    `reach` pixels away along them."""
    th = rng.uniform(0, np.pi, n)
    t = rng.uniform(-1, 1, n) * reach
    x = rng.uniform(-600, 600, n) + t * np.cos(th)
    y = rng.uniform(-340, 340, n) + t * np.sin(th)
    ls = np.log(np.stack([sigma * rng.uniform(0.6, 1.0, n), np.full(n, 0.05), np.full(n, 0.05)],
                         1) * z / f)
    return dict(means=np.stack([x * z / f, y * z / f, np.full(n, z) + 1e-3 * np.arange(n)],
                               1).astype(np.float32),
                log_scales=ls.astype(np.float32),
                quats=np.stack([np.cos(th / 2), 0 * th, 0 * th, np.sin(th / 2)],
                               1).astype(np.float32),
                opacity_logits=rng.uniform(-3, 3, n).astype(np.float32),
                sh=rng.uniform(-1, 1, (1, n, 3)).astype(np.float32), sh_degree=0)


NEEDLES = [(30, 60), (100, 200), (800, 1500), (3000, 700), (3000, 5000), (20000, 16000)]


@pytest.mark.parametrize("sigma,reach", NEEDLES)
@pytest.mark.parametrize("kw", [dict(pixels_per_thread_bwd=8),
                                dict(pixels_per_thread=2, pixels_per_thread_bwd=8),
                                dict(pixels_per_thread=8, tight_rect=False)])
def test_tile_kernels_leave_no_needle_out_either(sigma, reach, kw):
    """The masks of the tile kernels' warps: the bits of the block kernels."""
    rng = np.random.default_rng(sigma)
    p = _needles(rng, 300, sigma, reach)
    view = scenes.camera(1200, 680, 600.0, 600.0)
    gm = mapping.GaussianMap(p)
    out = []
    for k in (dict(tight_rect=kw.get("tight_rect", True)), dict(kw, deterministic=True)):
        rast = mapping.Rasterizer([view], gm.n, instance_capacity=1 << 20, **k)
        rast.forward(gm.gs_map())
        torch.cuda.synchronize()
        assert rast.counters().status == 0
        out.append([t.cpu().numpy() for t in (rast.images, rast.final_T, rast.last_idx)])
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("sigma,reach", [(100, 200), (800, 1500), (3000, 700), (3000, 5000),
                                         (20000, 16000)])
def test_long_needles_are_in_every_block_they_reach(sigma, reach):
    rng = np.random.default_rng(sigma + reach)
    p = _needles(rng, 300, sigma, reach)
    view = scenes.camera(1200, 680, 600.0, 600.0)
    gm = mapping.GaussianMap(p)
    dL = torch.tensor(rng.normal(size=(3, 680, 1200)).astype(np.float32)).cuda().reshape(-1)
    out = []
    for kw in (dict(), dict(deterministic=True, pixels_per_thread=8)):
        rast = mapping.Rasterizer([view], gm.n, instance_capacity=1 << 20, **kw)
        rast.forward(gm.gs_map())
        rast.render_bwd(gm.gs_map(), gm.gs_map_grad(), dL=dL)
        torch.cuda.synchronize()
        assert rast.counters().status == 0 and rast.counters().n_instances > 5000
        grad2d = rast.buffer(B.GS_BUF_GRAD2D, torch.float32)[:gm.n * 9].view(-1, 9)
        out.append([t.cpu().numpy() for t in (rast.images, rast.final_T, rast.last_idx, grad2d)])
    for x, y in zip(out[0][:3], out[1][:3]):
        np.testing.assert_array_equal(x, y)
    # (not dL/dmean: along a needle it is the difference of terms up to sigma times
    # as large, each a sum in FP32)
    for k in range(2, 9):
        assert U.rel_l2(out[0][3][:, k], out[1][3][:, k]) < 1e-5, k
