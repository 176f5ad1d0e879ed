"""A colour or a dL/dC that is not finite stays with the pixels that blend it: the
images, and the gradients of the Gaussians that share no pixel with it, are
what they are without it (up to the order of the float atomics)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2409_13055_gb300 import binding as B
from paper_2409_13055_gb300 import mapping, scenes

pytestmark = pytest.mark.gpu

SIZE = 64


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_13055_gb300 import build
    build.build()
    B.lib()


def _scene(channels):
    p, view = scenes.tiny_scene(300, SIZE, SIZE, seed=74, depth=(2.0, 3.0), log_scale=(-3.6, 0.3),
                                sh_degree=1)
    # some alphas past the clamp
    p["opacity_logits"] = np.random.default_rng(6).uniform(-2.0, 7.0, 300).astype(np.float32)
    return p, dict(view, channels=channels)


def _reach(p, view, tile):
    """[n, pixels]: where each Gaussian's alpha may count, a little widened."""
    proj = oracle.project(p, view, *tile)
    yy, xx = np.mgrid[0:SIZE, 0:SIZE]
    dx = proj["mean2d"][:, 0, None] - xx.ravel()
    dy = proj["mean2d"][:, 1, None] - yy.ravel()
    a, b, c = (proj["conic"][:, k, None] for k in range(3))
    alpha = proj["opacity"][:, None] * np.exp(-0.5 * (a * dx * dx + c * dy * dy) - b * dx * dy)
    return alpha >= 0.99 / 255.0, proj


def _run(p, view, tile, dL, **kw):
    gm = mapping.GaussianMap(p)
    rast = mapping.Rasterizer([view], gm.n, instance_capacity=1 << 18, tile=tile, **kw)
    rast.forward(gm.gs_map())
    rast.render_bwd(gm.gs_map(), gm.gs_map_grad(), dL=rast.pack([dL]))
    torch.cuda.synchronize()
    g = gm.grads()
    flat = [g[k].cpu().numpy().reshape(300, -1) for k in
            ("means", "log_scales", "quats", "opacity_logits")]
    flat += list(g["sh"].cpu().numpy())
    return rast.view_slice(rast.images, 0).cpu().numpy(), np.concatenate(flat, 1)


def _same(got, want):
    assert np.isfinite(got).all()
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)


@pytest.mark.parametrize("kw", [dict(), dict(density_stats=True)])
@pytest.mark.parametrize("channels", [3, 1])
@pytest.mark.parametrize("tile", [(8, 8), (16, 16)])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3e38])
def test_a_wild_colour_stays_with_its_pixels(tile, channels, kw, value):
    p, view = _scene(channels)
    reach, proj = _reach(p, view, tile)
    dL = np.random.default_rng(3).normal(size=(channels, SIZE, SIZE)).astype(np.float32)
    img0, grad0 = _run(p, view, tile, dL, **kw)
    g = int(np.argmin(np.hypot(*(proj["mean2d"] - 30.0).T) + 1e9 * (proj["tiles_touched"] == 0)))
    p["sh"][0, g] = value
    img, grad = _run(p, view, tile, dL, **kw)
    clear = ~reach[g]
    np.testing.assert_array_equal(img.reshape(channels, -1)[:, clear],
                                  img0.reshape(channels, -1)[:, clear])
    apart = ~(reach & reach[g]).any(1)
    # some of them lie in its blocks all the same
    r = proj["rect"][g]
    box = np.zeros((SIZE, SIZE), bool)
    box[r[1] * tile[1]:r[3] * tile[1], r[0] * tile[0]:r[2] * tile[0]] = True
    assert (apart & reach[:, box.ravel()].any(1)).sum() > 5
    _same(grad[apart], grad0[apart])


@pytest.mark.parametrize("channels", [3, 1])
@pytest.mark.parametrize("tile", [(8, 8), (16, 16)])
@pytest.mark.parametrize("value", [np.inf, np.nan, -3e38])
def test_a_wild_gradient_stays_with_its_pixel(tile, channels, value):
    p, view = _scene(channels)
    reach, _ = _reach(p, view, tile)
    dL = np.random.default_rng(4).normal(size=(channels, SIZE, SIZE)).astype(np.float32)
    _, grad0 = _run(p, view, tile, dL)
    dL[-1, 29, 31] = value
    _, grad = _run(p, view, tile, dL)
    apart = ~reach[:, 29 * SIZE + 31]
    assert (~apart).sum() > 0 and (apart & reach[:, 28 * SIZE + 27]).sum() > 0
    _same(grad[apart], grad0[apart])
