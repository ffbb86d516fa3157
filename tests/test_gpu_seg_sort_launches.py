"""The segment sort's launch by the mean list (one tile per CTA for long lists of a launch by
itself), and its test of a tile's pixels at every tile side: lists exactly as the binning
specification has them, and a stale saturation state's second visit equal to the waves."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    from paper_2606_18588_gb300 import splx as S
    c = S.Context()
    yield c
    c.close()


def test_long_lists_one_tile_per_cta(ctx):
    from test_gpu_seg_sort import test_mixed_lists_side_by_side as mixed_lists
    mixed_lists(ctx, 640, 480, 230)  # 4800 tiles of 230 keys, 300 keys or none among them


@pytest.mark.parametrize("tile", [8, 32])
def test_tiles_left_unsorted_by_a_stale_state(ctx, tile):
    from paper_2606_18588_gb300 import splx as S
    from paper_2606_18588_gb300.visibility import orders_for_views
    from gpu_util import subset_struct, to_device
    from test_oracle_pins import _cam, _saturating_slabs
    sc, off, boxes = _saturating_slabs(33)
    cams = [_cam(200, 150), _cam(131, 77)]
    orders = orders_for_views(boxes, cams)
    dev = to_device(sc)
    subs = [subset_struct(dev, int(off[k]), int(off[k + 1]), sc.sh_degree) for k in range(3)]
    out = []
    for stale in (False, True):
        b = S.Batch(ctx, subs, cams, S.opts(tile=tile))
        b.set_order(orders)
        if stale:
            planes = [torch.full((c.height * c.width,), 255, dtype=torch.uint8, device="cuda")
                      for c in cams]
            b.set_stale(planes)
        rgb = torch.empty(b.rgb_off[-1], device="cuda")
        T = torch.empty(b.total_pixels, device="cuda")
        for _ in range(2):
            b.forward(rgb, T)
        torch.cuda.synchronize()
        out.append((rgb, T, b.counters()["skipped_items"]))
        b.close()
    assert out[0][2] == out[1][2] > 0
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
