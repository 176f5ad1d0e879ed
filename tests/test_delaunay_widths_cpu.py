"""The triangulation's in-circle test in 64-bit integers (coordinates below
2^14) against the 128-bit one: moving every point by (2^14, 0) keeps their
order along the Z-curve and every predicate, so the triangles have to be the
same, one by one."""
import numpy as np
import pytest

from paper_2409_13055_gb300 import binding as B


@pytest.mark.parametrize("w,h,n", [(16384, 16384, 4000), (16384, 3, 2000), (40, 40, 1500),
                                   (2, 16384, 500), (752, 480, 6000)])
def test_both_widths_give_the_same_triangles(w, h, n):
    rng = np.random.default_rng(w + h)
    ids = rng.choice(w * h, min(n, w * h), replace=False)
    xy = np.stack([ids % w, ids // w], 1).astype(np.int32)
    xy[0] = (w - 1, h - 1) if (w - 1) + (h - 1) * w not in ids[1:] else xy[0]
    near = B.gs_delaunay(xy)
    far = B.gs_delaunay(xy + np.array([1 << 14, 0], np.int32))
    assert len(near) > n // 2
    np.testing.assert_array_equal(near, far)
