"""Projection and fill give a warp fewer Gaussians in small launches (32 down to 2): counts at
the edges of those steps, with rectangles of one tile and of hundreds, against the tile lists
of the binning specification, exactly."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_18588_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    from paper_2606_18588_gb300 import splx as S
    c = S.Context()
    yield c
    c.close()


@pytest.mark.parametrize("n", [1, 2, 3, 31, 9728, 9729, 19457, 38913, 77825, 155_649, 311_297])
def test_lists_at_every_gaussians_per_warp(ctx, n):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import subset_struct, to_device
    rng = np.random.default_rng(n)
    m = rng.uniform(-1.2, 1.2, (n, 3)).astype(np.float32)
    ls = rng.uniform(-6.0, -4.5, (n, 3)).astype(np.float32)
    ls[rng.integers(0, n, max(n // 200, 1))] = -1.5  # a few that reach hundreds of tiles
    sc = I.Scene(m, ls, rng.standard_normal((n, 4)).astype(np.float32),
                 rng.normal(0.0, 2.0, n).astype(np.float32),
                 np.zeros((n, 1, 3), np.float32), 0)
    cam = I.pinhole(333, 171, 150.0, (0.0, 0.0, -3.0), (0.0, 0.0, 0.0))
    p = S.new_partial(cam.height, cam.width)
    st = S.render_partial(ctx, subset_struct(to_device(sc), 0, n, 0), cam, S.opts(tile=16), p)
    ranges, keys, _ = st.export()
    vals = (keys & np.uint64(0xFFFFFFFF)).astype(np.uint32)
    start, lst = O.tile_lists(sc, cam, 16)
    assert np.array_equal(ranges[:, 1] - ranges[:, 0], np.diff(start).astype(ranges.dtype))
    for t in range(start.size - 1):
        a, b = int(start[t]), int(start[t + 1])
        ga, gb = int(ranges[t, 0]), int(ranges[t, 1])
        assert np.array_equal(vals[ga:gb], lst[a:b].astype(np.uint32)), t
    st.close()
