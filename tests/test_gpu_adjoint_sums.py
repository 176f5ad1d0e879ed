"""The pixel adjoint's sums over a block hold every bit of dL/dC: isolated
Gaussians, whose colour gradient is a weighted sum of dL/dC with weights that
the same map's gradient under dL/dC = 1 sums too.

The ratio of the two gradients against the one formed in FP64 from the rendered
weights: each side's products and sums round to nearest (up to 2^-24 each,
either way), so one ratio may be off by some 2^-22, but the mean over 3600 of
them by about 2^-24 / sqrt(3600) = 1e-9.  Operands cut to 22 bits would put it
near -2.5e-7 for the dL/dC used here, whose last two bits are ones; 2^-25 =
3e-8 is far from both."""
import numpy as np
import pytest
import torch

from paper_2409_13055_gb300 import binding as B
from paper_2409_13055_gb300 import mapping, scenes

pytestmark = pytest.mark.gpu

CELL, W, H = 16, 640, 480  # one Gaussian per cell of 16x16 pixels


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_13055_gb300 import build
    build.build()
    B.lib()


def _map(rng):
    gx, gy = np.meshgrid(np.arange(W // CELL), np.arange(H // CELL))
    n, f, z = gx.size, 500.0, 2.0
    px = gx.ravel() * CELL + 7.5 + rng.uniform(-1, 1, n)
    py = gy.ravel() * CELL + 7.5 + rng.uniform(-1, 1, n)
    view = scenes.camera(W, H, f, f)
    p = dict(means=np.stack([(px - view["cx"]) * z / f, (py - view["cy"]) * z / f,
                             np.full(n, z)], 1).astype(np.float32),
             # 1.4 to 1.6 pixels: alpha reaches 1/255 within 5.2 of the mean
             log_scales=np.log(rng.uniform(1.4, 1.6, (n, 3)) * z / f).astype(np.float32),
             quats=np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1)),
             opacity_logits=np.zeros(n, np.float32),
             sh=np.full((1, n, 3), 0.5 / 0.28209479177387814, np.float32), sh_degree=0)
    return p, view


@pytest.mark.parametrize("tile", [(8, 8), (16, 16)])
def test_colour_gradients_keep_the_last_bits_of_dL(tile):
    rng = np.random.default_rng(11)
    p, view = _map(rng)
    # in [1, 2), the last thirteen bits 1xxxxxxxxxx11
    bits = 0x3f800000 | (rng.integers(0, 1 << 10, (3, H, W)) << 13) | 0x1003 | \
        (rng.integers(0, 1 << 10, (3, H, W)) << 2)
    dL = bits.astype(np.uint32).view(np.float32)
    gm = mapping.GaussianMap(p)
    rast = mapping.Rasterizer([view], gm.n, instance_capacity=1 << 16, tile=tile)
    rast.forward(gm.gs_map())

    def colour_grads(d):
        rast.render_bwd(gm.gs_map(), gm.gs_map_grad(), dL=rast.pack([d]))
        torch.cuda.synchronize()
        return gm.grads()["sh"].cpu().numpy()[0].astype(np.float64)

    ones, got = colour_grads(np.ones_like(dL)), colour_grads(dL)
    w = rast.view_slice(rast.images, 0).cpu().numpy()[0].astype(np.float64)

    def cells(x):
        return x.reshape(H // CELL, CELL, W // CELL, CELL).sum((1, 3)).ravel()

    want = np.stack([cells(w * d.astype(np.float64)) for d in dL], 1) / cells(w)[:, None]
    err = got / ones / want - 1.0
    assert np.abs(err).max() < 2e-6
    assert abs(err.mean()) < 2.0 ** -25, err.mean()
