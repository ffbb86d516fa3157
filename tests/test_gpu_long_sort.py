"""The one-launch sort of long tile lists: lists that need no merge, one round and up to six
rounds in the same launch, with more (chunk, round) items than CTAs fit on the device, so that
items of different rounds and lists run side by side.  Orders are whole numbers: exact."""
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


@pytest.mark.parametrize("lengths", [(2049, 4097, 16385, 65536, 200_000), (2048, 2049), (40_961,)])
def test_mixed_list_lengths_in_one_launch(ctx, lengths):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import subset_struct, to_device
    rng = np.random.default_rng(len(lengths))
    cam = I.pinhole(16 * (len(lengths) + 1), 16, 60.0, (0.0, 0.0, -3.0), (0.0, 0.0, 0.0))
    parts = []
    for j, n in enumerate(lengths):  # list j: Gaussians around the centre of tile j
        z = rng.choice(np.float32([-0.5, -0.25, 0.0, 0.25]), n)  # equal depths: index order
        z += (rng.random(n) < 0.5) * rng.uniform(0.0, 0.2, n).astype(np.float32)
        px = 16 * j + 8 + rng.uniform(-1.0, 1.0, n)
        d = z + 3.0
        parts.append(np.stack([(px - cam.cx) / cam.fx * d, rng.uniform(-0.01, 0.01, n) * d, z], 1))
    m = np.concatenate(parts).astype(np.float32)
    m = m[rng.permutation(m.shape[0])]
    n = m.shape[0]
    sc = I.Scene(m, np.full((n, 3), -7.0, np.float32),
                 np.tile(np.float32([1, 0, 0, 0]), (n, 1)), np.zeros(n, np.float32),
                 np.zeros((n, 1, 3), np.float32), 0)
    start, lst = O.tile_lists(sc, cam, 16)
    assert sorted(np.diff(start))[-len(lengths):] == sorted(lengths)
    dev = to_device(sc)
    for _ in range(2):
        p = S.new_partial(cam.height, cam.width)
        st = S.render_partial(ctx, subset_struct(dev, 0, n, 0), cam, S.opts(tile=16), p)
        ranges, keys, _ = st.export()
        vals = (keys & np.uint64(0xFFFFFFFF)).astype(np.uint32)
        for t in range(start.size - 1):
            a, b = int(start[t]), int(start[t + 1])
            ga, gb = int(ranges[t, 0]), int(ranges[t, 1])
            assert gb - ga == b - a
            assert np.array_equal(vals[ga:gb], lst[a:b].astype(np.uint32)), t
        st.close()
