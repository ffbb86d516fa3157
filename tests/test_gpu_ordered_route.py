"""Saturation skipping in one forward launch: that the route is taken (fewer launches), with items
skipped at every tile side, and the same in a captured graph, whose kernels do not count."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("tile", [8, 16, 32])
def test_route_skips_what_the_waves_skip(tile):
    from paper_2606_18588_gb300 import splx as S
    from paper_2606_18588_gb300.visibility import orders_for_views
    from gpu_util import subset_struct, to_device
    from test_oracle_pins import _cam, _saturating_slabs
    ctx = S.Context()
    sc, off, boxes = _saturating_slabs(41)
    cams = [_cam(200, 150), _cam(131, 77)]
    dev = to_device(sc)
    b = S.Batch(ctx, [subset_struct(dev, int(off[k]), int(off[k + 1]), sc.sh_degree)
                      for k in range(3)], cams, S.opts(tile=tile))
    b.set_order(orders_for_views(boxes, cams))
    rgb = torch.empty(b.rgb_off[-1], device="cuda")
    T = torch.empty(b.total_pixels, device="cuda")

    def forward():
        rgb.fill_(float("nan"))
        n0 = ctx.launch_count
        b.forward(rgb, T)
        torch.cuda.synchronize()
        assert b.status()[0] == S.OK
        return rgb.clone(), T.clone(), b.counters()["skipped_items"], ctx.launch_count - n0

    c0, t0, skipped, waves = forward()
    b.tune_prefix_sort()
    c1, t1, skipped1, one = forward()
    # two view groups in waves: 3 x 2 x (sort, forward, the retries' sort and forward); one
    # sort, long sort and forward
    assert waves - one == 24 - 3
    assert skipped1 == skipped > 0
    assert torch.equal(c0, c1) and torch.equal(t0, t1)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        S.graph_begin(ctx, s)
        b.forward(rgb, T, stream=s)
        g = S.graph_end(ctx, s)
        for _ in range(2):
            rgb.fill_(float("nan"))
            g.launch(s)
    s.synchronize()
    assert torch.equal(rgb, c0) and torch.equal(T, t0)
    assert b.counters()["skipped_items"] == skipped  # the eager forward's
    g.close()
    b.close()
    ctx.close()
