"""The binning's routes: the one-launch depth sort of small plans and the
counting tile sort against the general radix sorts, at the edges of their
ranges.  All of them are exact: every buffer has to be equal."""
import numpy as np
import pytest
import torch

from paper_2409_13055_gb300 import binding as B
from paper_2409_13055_gb300 import mapping, scenes

pytestmark = pytest.mark.gpu

RADIX = (1 << 20) + 1  # an instance capacity past the counting sort's


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_13055_gb300 import build
    build.build()
    B.lib()


def _bins(p, views, capacity, **kw):
    """(counters, depth order, keys, values, ranges, image) of one binning; the
    depth order is checked against a stable sort of the projected depths."""
    gm = mapping.GaussianMap(p)
    rast = mapping.Rasterizer(views, gm.n, instance_capacity=capacity, **kw)
    rast.forward(gm.gs_map())
    c = rast.counters()
    vn = len(views) * gm.n
    touched = rast.buffer(B.GS_BUF_TOUCHED, torch.int32)[:vn].cpu().numpy()
    depth = rast.buffer(B.GS_BUF_PROJ, torch.float32)[:12 * vn].view(vn, 12)[:, 11].cpu().numpy()
    seen = np.nonzero(touched)[0]
    order = rast.buffer(B.GS_BUF_DEPTH_ORDER, torch.int32)[:len(seen)].cpu().numpy()
    np.testing.assert_array_equal(order, seen[np.argsort(depth[seen], kind="stable")])
    assert c.n_instances_raw == touched.astype(np.int64).sum()
    n = int(c.n_instances)
    keys, vals = (rast.buffer(b, torch.int32)[:n].cpu().numpy()
                  for b in (B.GS_BUF_TILE_KEYS, B.GS_BUF_TILE_VALUES))
    ranges = rast.buffer(B.GS_BUF_RANGES, torch.int32)[:2 * rast.total_tiles].cpu().numpy()
    assert (np.diff(keys) >= 0).all()
    return (c.status, n, c.n_instances_raw), keys, vals, ranges, rast.images.cpu().numpy()


def _same(p, views, capacity=1 << 20, **kw):
    a, b = _bins(p, views, capacity, **kw), _bins(p, views, RADIX, **kw)
    assert a[0] == b[0]
    for x, y in zip(a[1:], b[1:]):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("n", [1, 31, 1025, 32768, 32769, 131072, 131073])
def test_pairs_at_the_edges_of_the_depth_sorts(n):
    _same(scenes.room_scene(n, seed=81, sh_degree=0), [scenes.camera(200, 120, 120.0, 120.0)])


@pytest.mark.parametrize("tile,size", [((8, 8), (8, 8)), ((8, 8), (1237, 1200)),
                                       ((8, 8), (1240, 1240)), ((16, 16), (97, 61))])
def test_tiles_at_the_edges_of_the_counting_sort(tile, size):
    """One tile, just under and over the 24000 it takes, ragged images."""
    w, h = size
    _same(scenes.room_scene(3000, seed=82, sh_degree=0), [scenes.camera(w, h, 0.6 * w, 0.6 * w)],
          tile=tile)


def test_views_tall_boxes_and_square_rects():
    p = scenes.room_scene(5000, seed=83, sh_degree=0)
    p["log_scales"][::50] += 3.5  # boxes of hundreds of tiles, taller than 16 rows
    R, t = scenes.random_pose(np.random.default_rng(1), 0.3, 20.0)
    views = [scenes.camera(320, 240, 200.0, 200.0), scenes.camera(209, 133, 130.0, 130.0, channels=1),
             scenes.camera(320, 240, 200.0, 200.0, R=R, t=t)]
    for tight in (True, False):
        _same(p, views, tile=(8, 8), tight_rect=tight)


def test_ties_far_depths_and_nothing_visible():
    p = scenes.room_scene(4000, seed=84, sh_degree=0)
    view = [scenes.camera(160, 120, 100.0, 100.0)]
    flat = dict(p, means=p["means"].copy())
    flat["means"][:, 2] = 2.0  # one depth for all: the index decides
    _same(flat, view)
    far = dict(p, means=p["means"] * np.geomspace(1e-3, 1e5, 4000)[:, None].astype(np.float32))
    far["log_scales"] = p["log_scales"] + np.log(np.geomspace(1e-3, 1e5, 4000))[:, None].astype(
        np.float32)
    _same(far, view, near_z=1e-4)  # keys of more than 27 bits
    _same(p, [scenes.camera(160, 120, 100.0, 100.0, t=[0.0, 0.0, -50.0])])


def test_instances_past_the_capacity_are_the_last_emitted():
    """The surplus is dropped in depth order: a capped binning lists, tile by
    tile, the instances of the full one whose emission position is below the
    capacity."""
    p = scenes.room_scene(6000, seed=85, sh_degree=0)
    view = [scenes.camera(200, 150, 120.0, 120.0)]
    full = _bins(p, view, 1 << 20)
    cap = full[0][1] // 3
    status, keys, vals, ranges, _ = _bins(p, view, cap)
    assert status == (B.GS_DEV_CAPACITY, cap, full[0][1])
    lists = {t: full[2][a:b].tolist() for t, (a, b) in enumerate(full[3].reshape(-1, 2))}
    for t, (a, b) in enumerate(ranges.reshape(-1, 2)):
        assert vals[a:b].tolist() == lists[t][:b - a]


def test_deterministic_plan_is_the_same_on_both_routes():
    p = scenes.room_scene(3000, seed=86, sh_degree=1)
    view = scenes.camera(160, 120, 100.0, 100.0)
    gm = mapping.GaussianMap(p)
    out = []
    for capacity in (1 << 20, RADIX):
        rast = mapping.Rasterizer([view], gm.n, instance_capacity=capacity, tile=(8, 8),
                                  pixels_per_thread_bwd=2, deterministic=True)
        rast.forward(gm.gs_map())
        rast.render_bwd(gm.gs_map(), gm.gs_map_grad(), dL=torch.ones_like(rast.dL))
        out.append([rast.images.cpu().numpy(), gm.grad.cpu().numpy()])
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)
