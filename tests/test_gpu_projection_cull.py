"""The projection's cheap test of what cannot reach an image, against the oracle
where the answer is close: Gaussians whose box ends within a few pixels of an
image's edge, and around the near plane.  Whole numbers: all of them equal
outside the oracle's guard bands."""
import numpy as np
import pytest
import torch

import oracle
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


def _edge_scene(view, n, seed, zmax):
    """Isotropic and flat Gaussians around the borders of the view's image."""
    rng = np.random.default_rng(seed)
    f, w, h = view["fx"], view["width"], view["height"]
    z = np.exp(rng.uniform(np.log(0.1), np.log(zmax), n))
    z[::16] = 0.2 * (1 + rng.uniform(-1, 1, len(z[::16])) * 10.0 ** rng.integers(-7, 1, len(z[::16])))
    s = z / f * np.exp(rng.uniform(np.log(0.05), np.log(400.0), n))
    ls = np.log(np.stack([s, s * rng.choice([1.0, 0.01], n), s * rng.choice([1.0, 0.01], n)], 1))
    r = 3 * s * f / z + 1
    mx, my = rng.uniform(-0.2 * w, 1.2 * w, n), rng.uniform(-0.2 * h, 1.2 * h, n)
    side, off = rng.integers(0, 5, n), rng.uniform(-8, 8, n)
    mx = np.where(side == 0, -r + off, np.where(side == 1, w + r + off, mx))
    my = np.where(side == 2, -r + off, np.where(side == 3, h + r + off, my))
    cam = np.stack([(mx - view["cx"]) / f * z, (my - view["cy"]) / view["fy"] * z, z], 1)
    R, t = np.asarray(view["R"], np.float64), np.asarray(view["t"], np.float64)
    means = (cam - t) @ R
    q = rng.normal(size=(n, 4))
    p = dict(scenes.tiny_scene(n, w, h, seed=seed, sh_degree=0)[0])
    p.update(means=means.astype(np.float32), log_scales=ls.astype(np.float32),
             quats=(q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
             opacity_logits=rng.uniform(-1, 4, n).astype(np.float32))
    return p


@pytest.mark.parametrize("zmax,centre", [(5.0, (0.5, 0.5)), (400.0, (0.1, 0.8)), (20.0, (-0.3, 1.4))])
@pytest.mark.parametrize("tight", [False, True])
def test_boxes_that_end_near_an_edge(zmax, centre, tight):
    w, h = 203, 117
    R, t = scenes.random_pose(np.random.default_rng(9), 0.4, 60.0)
    view = scenes.camera(w, h, 150.0, 170.0, centre[0] * w, centre[1] * h, R=R, t=t)
    p = _edge_scene(view, 6000, 91, zmax)
    gm = mapping.GaussianMap(p)
    rast = mapping.Rasterizer([view], gm.n, instance_capacity=1 << 21, tile=(8, 8), tight_rect=tight)
    rast.forward(gm.gs_map())
    torch.cuda.synchronize()
    g = U.gpu_projection(rast, gm.n)
    o = oracle.project(p, view, 8, 8, tight=tight)
    ok = (o["guard"] & U.FWD_GUARDS) == 0
    assert ok.mean() > 0.95
    np.testing.assert_array_equal(g["touched"][ok], o["tiles_touched"][ok])
    vis = ok & (o["tiles_touched"] > 0)
    assert 500 < vis.sum() < 5900
    np.testing.assert_array_equal(g["radius"][vis], o["radius"][vis])
    np.testing.assert_array_equal(g["rect"][vis], o["rect"][vis])
