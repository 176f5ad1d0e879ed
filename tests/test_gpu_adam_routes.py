"""The vectorised Adam kernels, which write nothing where state and gradient are
all zero and take planes off the 16-byte grid by float4 of the buffer, against
the float-by-float kernels (buffers off the 16-byte grid), bit for bit."""
import numpy as np
import pytest
import torch

from paper_2409_13055_gb300 import binding as B
from paper_2409_13055_gb300 import mapping

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_13055_gb300 import build
    build.build()
    B.lib()


def _state(n, degree, seed):
    """(offsets, total, p, g, m, v, group_vis): about half of the groups of 32
    never reached, some moments -0, some gradients zero with moments."""
    off, total = mapping.param_layout(n, degree)
    rng = np.random.default_rng(seed)
    p, g, m, v = (rng.normal(size=total).astype(np.float32) for _ in range(4))
    v = np.abs(v)
    seen = rng.uniform(size=(n + 31) // 32) < 0.5
    K = (degree + 1) ** 2
    planes = [(off["means"], 3), (off["log_scales"], 3), (off["quats"], 4),
              (off["opacity_logits"], 1)] + [(off["sh"] + 3 * n * k, 3) for k in range(K)]
    used = np.zeros(total, bool)
    for start, s in planes:
        own = np.repeat(np.repeat(seen, 32)[:n], s)
        cut = slice(start, start + s * n)
        used[cut] = True
        for a in (g, m, v):
            a[cut] *= own
        m[cut] = np.where(rng.uniform(size=s * n) < 0.02, np.float32(-0.0), m[cut])
        g[cut] *= rng.uniform(size=s * n) < 0.8
    for a in (p, g, m, v):
        a[~used] = 0.0
    return off, total, p, g, m, v, seen.astype(np.uint8)


def _run(state, shift, grouped, n, lr, eps):
    off, total, p, g, m, v, vis = state
    bufs = []
    for a in (p, g, m, v):
        b = torch.zeros(total + 4, device="cuda")
        b[shift:shift + total] = torch.from_numpy(a).cuda()
        bufs.append(b[shift:shift + total])
    step = torch.full((1,), 6, dtype=torch.int32, device="cuda")
    starts = [off[k] for k in mapping.GROUPS] + [total]
    starts[0] = 0
    if grouped:
        B.gs_adam_step_groups(*bufs, starts, lr, mapping.GROUP_STRIDES, n,
                              torch.from_numpy(vis).cuda(), 0.9, 0.999, eps, step)
    else:
        B.gs_adam_step(*bufs, starts, lr, 0.9, 0.999, eps, step)
    assert int(step.item()) == 7
    return [b.cpu().numpy().view(np.uint32) for b in (bufs[0], bufs[2], bufs[3])]


LR = [1.6e-4, 5e-3, 1e-3, 0.05, 2.5e-3, 1.25e-4]


@pytest.mark.parametrize("n,degree", [(1, 0), (2, 1), (5, 0), (33, 3), (1000, 2), (1003, 3),
                                      (103_790, 0), (103_793, 1), (450_001, 0)])
def test_vector_and_scalar_steps_agree(n, degree):
    state = _state(n, degree, n)
    # (below five Gaussians a group's padding holds more planes than the grouped
    # step takes: refused, as it was)
    for grouped in (False, True) if n >= 5 else (False,):
        for x, y in zip(_run(state, 0, grouped, n, LR, 1e-15), _run(state, 1, grouped, n, LR, 1e-15)):
            np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("lr,eps", [([float("inf")] + LR[1:], 1e-15), (LR, 0.0), ([0.0] * 6, 1e-8)])
def test_rates_and_eps_that_do_change_idle_floats(lr, eps):
    """An infinite rate or eps = 0 turns an idle parameter into NaN: as before."""
    state = _state(1003, 1, 9)
    for grouped in (False, True):
        for x, y in zip(_run(state, 0, grouped, 1003, lr, eps), _run(state, 1, grouped, 1003, lr, eps)):
            nan = np.isnan(x.view(np.float32))
            np.testing.assert_array_equal(nan, np.isnan(y.view(np.float32)))
            np.testing.assert_array_equal(x[~nan], y[~nan])
