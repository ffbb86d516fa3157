"""The tile segments' sort with several tiles per CTA (eight for short lists, two for long
ones): lists around the warp's 256 keys, the CTA's 2048 and beyond side by side, exactly; and
saturation-skipping waves over such launches leave a depth-separated scene unchanged."""
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


LENGTHS = [0, 1, 2, 255, 256, 257, 2047, 2048, 2049, 4097, 8, 300, 0, 700, 1, 9, 33]


@pytest.mark.parametrize("W,H,fill", [(1024, 960, 0), (640, 480, 140)])
def test_mixed_lists_side_by_side(ctx, W, H, fill):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import subset_struct, to_device
    rng = np.random.default_rng(W)
    cam = I.pinhole(W, H, 400.0, (0.0, 0.0, -3.0), (0.0, 0.0, 0.0))
    tx = (W + 7) // 8
    nt = tx * ((H + 7) // 8)
    count = np.full(nt, fill)
    for r in range(3):  # three runs of the lengths, at offsets that are no multiple of eight
        count[1000 * r + 3:1000 * r + 3 + len(LENGTHS)] = LENGTHS
    tile = np.repeat(np.arange(nt), count)
    n = tile.size
    z = rng.choice(np.float32([-0.5, 0.0, 0.25]), n) + rng.integers(0, 5, n) * 0.01
    d = z + 3.0
    px = 8 * (tile % tx) + 4 + rng.uniform(-0.5, 0.5, n)
    py = 8 * (tile // tx) + 4 + rng.uniform(-0.5, 0.5, n)
    m = np.stack([(px - cam.cx) / cam.fx * d, (py - cam.cy) / cam.fy * d, z], 1)
    m = m.astype(np.float32)[rng.permutation(n)]
    sc = I.Scene(m, np.full((n, 3), -8.0, np.float32),
                 np.tile(np.float32([1, 0, 0, 0]), (n, 1)), np.zeros(n, np.float32),
                 np.zeros((n, 1, 3), np.float32), 0)
    start, lst = O.tile_lists(sc, cam, 8)
    assert np.array_equal(np.diff(start), count)
    p = S.new_partial(H, W)
    st = S.render_partial(ctx, subset_struct(to_device(sc), 0, n, 0), cam, S.opts(tile=8), p)
    ranges, keys, _ = st.export()
    vals = (keys & np.uint64(0xFFFFFFFF)).astype(np.uint32)
    assert np.array_equal(ranges[:, 1] - ranges[:, 0], count.astype(ranges.dtype))
    order = np.concatenate([vals[a:b] for a, b in ranges.astype(np.int64) if b > a])
    assert np.array_equal(order, lst.astype(np.uint32))
    st.close()


@pytest.mark.parametrize("size", [(512, 480), (1100, 1000)])
def test_waves_over_grouped_tiles(ctx, size):
    from paper_2606_18588_gb300 import splx as S
    from paper_2606_18588_gb300.visibility import orders_for_views
    from gpu_util import subset_struct, to_device
    from test_oracle_pins import _cam, _saturating_slabs
    sc, off, boxes = _saturating_slabs(21)
    cams = [_cam(*size)]
    dev = to_device(sc)
    subs = [subset_struct(dev, int(off[k]), int(off[k + 1]), sc.sh_degree)
            for k in range(len(off) - 1)]
    out = []
    for order in (orders_for_views(boxes, cams), None):
        b = S.Batch(ctx, subs, cams, S.opts(tile=8))
        b.set_order(order)
        rgb = torch.empty(b.rgb_off[-1], device="cuda")
        b.forward(rgb)
        torch.cuda.synchronize()
        out.append((rgb, b.counters()["skipped_items"]))
        b.close()
    assert out[0][1] > 0 and out[1][1] == 0
    assert torch.equal(out[0][0], out[1][0])
