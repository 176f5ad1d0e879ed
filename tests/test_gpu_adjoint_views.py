"""The projection adjoint of plans of several views, at the edges of its warps and
CTAs: adding to gradients gives the bits of the gradients alone plus what was
there, and the grouped form those of the plain one."""
import numpy as np
import pytest
import torch

from paper_2409_13055_gb300 import binding as B
from paper_2409_13055_gb300 import mapping, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_13055_gb300 import build
    build.build()
    B.lib()


GROUPS = ("means", "log_scales", "quats", "opacity_logits", "sh")


def _grads(gm, fill):
    g = torch.Generator(device="cuda").manual_seed(3)
    out = []
    for name in GROUPS:
        t = gm._views(gm.data)[name]
        out.append(torch.randn(t.shape, device="cuda", generator=g) if fill == "random"
                   else torch.full_like(t, fill))
    return out


def _ptr(g):
    return B.gs_map_grad(*[t.data_ptr() for t in g])


@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 4999])
@pytest.mark.parametrize("degree", [0, 1, 2, 3])
@pytest.mark.parametrize("odd", [None, "overflow", "nan"])
def test_adding_is_the_sum_bit_for_bit(n, degree, odd):
    p = scenes.room_scene(n, seed=61, sh_degree=degree)
    p["means"][n // 2:, 2] -= 50.0  # behind every camera: not touched
    if odd == "overflow":
        p["log_scales"][n - 1] = 60.0
    elif odd == "nan":
        p["means"][n - 1, 0] = np.nan
    R, t = scenes.random_pose(np.random.default_rng(2), 0.2, 15.0)
    views = [scenes.camera(96, 64, 60.0, 60.0), scenes.camera(80, 72, 55.0, 55.0, channels=1),
             scenes.camera(96, 64, 60.0, 60.0, R=R, t=t)]
    gm = mapping.GaussianMap(p)
    rast = mapping.Rasterizer(views, gm.n, instance_capacity=1 << 20)
    m = gm.gs_map()
    rast.forward(m)
    rast.loss_l1_ssim(torch.rand_like(rast.images), 0.2)
    rast.render_bwd_pixels()
    alone, base, added = _grads(gm, float("nan")), _grads(gm, "random"), _grads(gm, "random")
    rast.project_bwd(m, _ptr(alone))
    rast.project_bwd(m, _ptr(added), accumulate=True)
    grouped = _grads(gm, 7.0)
    vis = torch.full(((n + 31) // 32,), 9, dtype=torch.uint8, device="cuda")
    rast.project_bwd_groups(m, _ptr(grouped), vis)
    torch.cuda.synchronize()
    seen = rast.buffer(B.GS_BUF_TOUCHED, torch.int32)[:3 * n].view(3, n).ne(0).any(0).cpu().numpy()
    assert n < 100 or 0 < seen.sum() < n
    pad = np.zeros(len(vis) * 32, bool)
    pad[:n] = seen
    want_vis = pad.reshape(-1, 32).any(1)
    np.testing.assert_array_equal(vis.cpu().numpy(), want_vis)
    written = np.repeat(want_vis, 32)[:n]
    for name, a, b, c, d in zip(GROUPS, alone, base, added, grouped):
        a, b, c, d = (x.cpu().numpy() for x in (a, b, c, d))
        np.testing.assert_array_equal(c, a + b, err_msg=name)
        axis = 1 if name == "sh" else 0
        np.testing.assert_array_equal(np.compress(written, d, axis), np.compress(written, a, axis))
        assert (np.compress(~written, d, axis) == 7.0).all()
        if odd is None:
            assert np.isfinite(a).all()
            assert (np.compress(~seen, a, axis) == 0.0).all()
