"""Saturation skipping in one forward launch (a CTA renders a tile's subsets front to back),
which a batch takes once the tuning has found that its long lists are walked to their ends or
that little is skipped: images, transmittances, skipped items and gradients equal those of
the waves, on a scene one side of which saturates behind a wall and the other never does."""
import numpy as np
import pytest

from paper_2606_18588_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    from paper_2606_18588_gb300 import splx as S
    c = S.Context()
    yield c
    c.close()


def _scene(wall_on):
    # faint Gaussians in depth, and a wall of opaque ones in front of the left half; without
    # it fewer of them, so that no list is long and nothing is skipped
    sc = I.uniform_scene(40_000 if wall_on else 4_000, 72, 1, log_scale_mu=-3.5)
    sc.opacity_logits[:] = sc.opacity_logits - 2.5
    rng = np.random.default_rng(5)
    n = 4_000
    m = np.stack([rng.uniform(-1.4, -0.2, n), rng.uniform(-1.2, 1.2, n),
                  rng.uniform(-1.3, -1.2, n)], 1).astype(np.float32)
    wall = I.Scene(m, np.full((n, 3), -2.2, np.float32),
                   np.tile(np.float32([1, 0, 0, 0]), (n, 1)), np.full(n, 4.0, np.float32),
                   rng.normal(0.0, 0.3, (n, 4, 3)).astype(np.float32), 1)
    if wall_on:
        sc = I.Scene(*[np.concatenate([a, b]) for a, b in zip(sc.arrays(), wall.arrays())], 1)
    perm, off, boxes = I.kd_partition(sc.means, 4)
    return sc.take(perm), off, boxes


@pytest.mark.parametrize("wall", [True, False])
@pytest.mark.parametrize("tile", [8, 16, 32])
def test_one_launch_equals_the_waves(ctx, tile, wall):
    from paper_2606_18588_gb300 import splx as S
    from paper_2606_18588_gb300.visibility import orders_for_views
    from gpu_util import params_struct, rel_l2, subset_struct, to_device, zeros_like_params
    sc, off, boxes = _scene(wall)
    cams = [I.pinhole(64, 64, 60.0, (0.0, 0.0, -3.0), (0, 0, 0)),
            I.pinhole(83, 45, 50.0, (0.2, -0.1, -3.2), (0, 0, 0))]
    dev = to_device(sc)
    K = len(off) - 1
    subs = [subset_struct(dev, int(off[k]), int(off[k + 1]), 1) for k in range(K)]
    b = S.Batch(ctx, subs, cams, S.opts(tile=tile))
    b.set_order(orders_for_views(boxes, cams))
    dL = torch.from_numpy(np.random.default_rng(1).standard_normal(
        b.rgb_off[-1]).astype(np.float32)).cuda()
    res = []
    for tuned in (False, True):
        if tuned:
            b.tune_prefix_sort()
        rgb = torch.empty(b.rgb_off[-1], device="cuda")
        T = torch.empty(b.total_pixels, device="cuda")
        g = zeros_like_params(dev)
        for _ in range(2):  # a second forward must not see the first one's leftovers
            b.forward(rgb, T)
        b.backward(dL, None, [params_struct(g, int(off[k]), int(off[k + 1]), 1)
                              for k in range(K)])
        torch.cuda.synchronize()
        assert b.status()[0] == S.OK
        res.append((rgb, T, g, b.counters()))
    (rgb0, T0, g0, c0), (rgb1, T1, g1, c1) = res
    if wall and tile != 8:  # (8x8 tiles have no list beyond a prefix here)
        assert c0["prefix_items"] > 0 and c1["prefix_items"] == 0
    assert c0["skipped_items"] == c1["skipped_items"]
    assert c0["skipped_items"] > 0 or tile == 32 or not wall  # (no whole 32x32 tile lies behind the wall)
    assert torch.equal(rgb0, rgb1) and torch.equal(T0, T1)
    for k in g0:
        assert rel_l2(g1[k].cpu().numpy(), g0[k].cpu().numpy()) < 1e-5, k
    b.close()
