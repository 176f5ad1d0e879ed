"""The tile kernels (a warp or a CTA per tile), at the tiles that are not whole 8x8
blocks and in the deterministic adjoint of larger tiles: every number of pixels
per thread and several batches, both channel counts, square and tight lists,
with and without the density statistic, forward and backward against the FP64
oracle within the tolerances of test_gpu_blocks.py."""
import numpy as np
import pytest
import torch

from paper_2409_13055_gb300 import binding as B
from paper_2409_13055_gb300 import mapping, scenes
from tests import gpu_util as U
from tests.test_gpu_blocks import _check

pytestmark = pytest.mark.gpu

TILES = {(16, 4): (1, 2), (4, 16): (1, 2), (64, 4): (1, 2, 4, 8), (4, 64): (1, 2, 4),
         (2, 32): (1, 2), (128, 2): (1, 8)}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_13055_gb300 import build
    build.build()
    B.lib()


def _scene(channels, n=900):
    p, view = scenes.tiny_scene(n, 97, 61, seed=71, sh_degree=1)
    return p, dict(view, channels=channels)


@pytest.mark.parametrize("tight", [True, False])
@pytest.mark.parametrize("channels", [3, 1])
@pytest.mark.parametrize("tile,ppt", [(t, q) for t in TILES for q in TILES[t]])
def test_parity_at_tiles_that_are_not_blocks(tile, ppt, channels, tight):
    p, view = _scene(channels)
    _check(p, view, tile, tight_rect=tight, pixels_per_thread=ppt,
           smem_batch={1: 256, 2: 128, 4: 64, 8: 32}[ppt], density_stats=channels == 3)


def _render(p, view, tile, dL, **kw):
    gm = mapping.GaussianMap(p)
    rast = mapping.Rasterizer([view], gm.n, instance_capacity=1 << 20, tile=tile,
                              bg=(0.1, 0.2, 0.3), **kw)
    rast.forward(gm.gs_map())
    rast.render_bwd(gm.gs_map(), gm.gs_map_grad(), dL=dL)
    torch.cuda.synchronize()
    assert rast.counters().status == 0
    out = [t.cpu().numpy() for t in (rast.images, rast.final_T, rast.last_idx, gm.grad)]
    if kw.get("density_stats"):
        out.append(rast.buffer(B.GS_BUF_ABSGRAD, torch.float32)[:2 * gm.n].cpu().numpy())
    return out


@pytest.mark.parametrize("channels", [3, 1])
@pytest.mark.parametrize("tile", list(TILES))
def test_pixels_per_thread_and_batches_change_no_bit(tile, channels):
    """Images, transmittance and last_idx bit for bit, gradients up to the order of
    their sums (1e-5, as in test_gpu_parity.py)."""
    p, view = _scene(channels)
    rng = np.random.default_rng(9)
    dL = torch.tensor(rng.normal(size=channels * 97 * 61).astype(np.float32)).cuda()
    ref = _render(p, view, tile, dL, smem_batch=32)
    for ppt in TILES[tile]:
        for batch in (64, 256):
            got = _render(p, view, tile, dL, smem_batch=batch, pixels_per_thread=ppt)
            for x, y in zip(got[:3], ref[:3]):
                np.testing.assert_array_equal(x, y)
            assert U.rel_l2(got[3], ref[3]) < 1e-5, (ppt, batch)


@pytest.mark.parametrize("channels", [3, 1])
@pytest.mark.parametrize("tile,ppt", [((16, 16), 8), ((32, 8), 8), ((16, 8), 4), ((16, 4), 2),
                                      ((4, 16), 2), ((64, 4), 8)])
def test_deterministic_adjoint_of_every_tile(tile, ppt, channels):
    p, view = _scene(channels)
    _check(p, view, tile, deterministic=True, pixels_per_thread_bwd=ppt)
    rng = np.random.default_rng(10)
    dL = torch.tensor(rng.normal(size=channels * 97 * 61).astype(np.float32)).cuda()
    det = dict(deterministic=True, pixels_per_thread_bwd=ppt, density_stats=True)
    runs = [_render(p, view, tile, dL, **det, smem_batch_bwd=b) for b in (32, 128, 32)]
    for got in runs[1:]:
        for x, y in zip(got, runs[0]):
            np.testing.assert_array_equal(x, y)
    atomic = _render(p, view, tile, dL, density_stats=True)
    for x, y in zip(runs[0][:3], atomic[:3]):
        np.testing.assert_array_equal(x, y)
    assert U.rel_l2(runs[0][3], atomic[3]) < 1e-5
    # sums of magnitudes: some ten roundings of 2^-24 each way
    assert U.rel_l2(runs[0][4], atomic[4]) < 1e-6
