"""The radix passes of larger plans at the edges of their digits and blocks: the
depth order against a stable sort of the projected depths, the instances against
the order (tile, depth, index).  Whole numbers: everything equal."""
import numpy as np
import pytest
import torch

from paper_2409_13055_gb300 import binding as B
from paper_2409_13055_gb300 import mapping, scenes

pytestmark = pytest.mark.gpu

BIG = (1 << 20) + 1  # an instance capacity of the radix route


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_13055_gb300 import build
    build.build()
    B.lib()


def _check(p, view, **kw):
    gm = mapping.GaussianMap(p)
    rast = mapping.Rasterizer([view], gm.n, instance_capacity=BIG, **kw)
    m = gm.gs_map()
    rast.project(m)
    rast.bin_sort(gm.n)
    rast.bin_sort(gm.n)  # (a second binning of the same projection)
    torch.cuda.synchronize()
    c = rast.counters()
    assert c.status == 0
    touched = rast.buffer(B.GS_BUF_TOUCHED, torch.int32)[:gm.n].cpu().numpy()
    depth = rast.buffer(B.GS_BUF_PROJ, torch.float32)[:12 * gm.n].view(gm.n, 12)[:, 11].cpu().numpy()
    seen = np.nonzero(touched)[0]
    order = rast.buffer(B.GS_BUF_DEPTH_ORDER, torch.int32)[:len(seen)].cpu().numpy()
    np.testing.assert_array_equal(order, seen[np.argsort(depth[seen], kind="stable")])
    n = int(c.n_instances)
    assert n == touched.astype(np.int64).sum()
    keys, vals = (rast.buffer(b, torch.int32)[:n].cpu().numpy()
                  for b in (B.GS_BUF_TILE_KEYS, B.GS_BUF_TILE_VALUES))
    np.testing.assert_array_equal(np.lexsort((vals, depth[vals], keys)), np.arange(n))
    np.testing.assert_array_equal(np.bincount(vals, minlength=gm.n), touched)
    ranges = rast.buffer(B.GS_BUF_RANGES, torch.int32)[:2 * rast.total_tiles].cpu().numpy()
    lengths = np.bincount(keys, minlength=rast.total_tiles)
    np.testing.assert_array_equal(ranges[1::2] - ranges[::2], lengths)
    return len(seen)


def _line(n, z):
    """n small Gaussians on the optical axis at depths z."""
    p = scenes.room_scene(n, seed=71, sh_degree=0)
    p["means"][:] = 0.0
    p["means"][:, 2] = z
    p["log_scales"][:] = -40.0
    p["opacity_logits"][:] = 1.0
    return p


@pytest.mark.parametrize("n", [131073, 200_000, (1 << 20) - 1, 1 << 20])
def test_pairs_at_the_edges_of_the_blocks(n):
    p = scenes.room_scene(n, seed=72, sh_degree=0)
    p["log_scales"] -= 1.0
    assert _check(p, scenes.camera(64, 48, 30.0, 30.0)) > n // 20


@pytest.mark.parametrize("near,far", [(0.2, 0.2000001), (0.2, 0.21), (0.2, 50.0), (1e-3, 1e3),
                                      (1e-30, 1e30)])
def test_depths_of_one_to_thirty_one_bits(near, far):
    """The digits follow the largest depth; ties keep their index order."""
    n = 150_000
    rng = np.random.default_rng(73)
    z = np.exp(rng.uniform(np.log(near), np.log(far), n)).astype(np.float32)
    z = np.maximum(z, np.nextafter(np.float32(near), np.float32(np.inf)))
    z[::7] = z[0]
    # (boxes of the nearest of them overflow at 1e-30: culled)
    assert _check(_line(n, z), scenes.camera(16, 16, 8.0, 8.0), near_z=near) > 0.9 * n


@pytest.mark.parametrize("w,h", [(256, 256), (264, 256), (5792, 5792), (8192, 8192), (8200, 8192)])
def test_tiles_of_one_two_and_three_digits(w, h):
    """1024 tiles (one digit of ten bits), 1056 (two of six), ~2^19, 2^20 (two of
    ten) and a few more (three of seven)."""
    p = scenes.room_scene(150_000, seed=74, sh_degree=0)
    p["log_scales"] -= np.float32(np.log(max(w / 256.0, 1.0)))
    assert _check(p, scenes.camera(w, h, 0.6 * w, 0.6 * w), tile=(8, 8)) > 1000
