"""What splx_batch_tune_prefix_sort decides: a stale saturation state, an eager forward made
before the subset orders were set and persistent CTAs leave the selected prefixes on (there are
no waves to replace, or none were counted); one forward launch instead of the waves is given up
when cameras, orders or the launch form change, and weighed again by the next call."""
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


CAM = I.pinhole(256, 192, 60.0, (0.06, 0.06, -3.0), (0.06, 0.06, 0.0))
ORDER = np.array([[0, 1]])


def _open_scene(clump=4_000):
    """Faint Gaussians everywhere, which saturate nothing, in two subsets (near and far), and
    opaque ones over one tile (128-143, 96-111) in the far subset: one list that a selected
    prefix serves."""
    rng = np.random.default_rng(4)
    n = 2_000
    faint = I.uniform_scene(n, 61, 0, log_scale_mu=-4.0)
    faint.opacity_logits[:] = -3.0
    c = I.uniform_scene(clump, 62, 0, log_scale_mu=-4.0, log_scale_sigma=0.1)
    px = np.stack([rng.uniform(126, 146, clump), rng.uniform(94, 114, clump)], 1)
    z = rng.uniform(0.5, 0.9, clump)
    c.means[:, :2] = (px - [CAM.cx, CAM.cy]) / CAM.fx * (z + 3.0)[:, None] + CAM.eye[:2]
    c.means[:, 2] = z
    c.opacity_logits[:] = 3.0
    near = np.flatnonzero(faint.means[:, 2] < 0.0)
    far = np.flatnonzero(faint.means[:, 2] >= 0.0)
    perm = np.concatenate([near, far, np.arange(n, n + clump)])
    sc = I.Scene(*[np.concatenate([a, b]) for a, b in zip(faint.arrays(), c.arrays())], 0)
    return sc.take(perm), np.array([0, near.size, n + clump])


def _batch(ctx, sc, off, cam=CAM, capacity=1 << 20):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import subset_struct, to_device
    dev = to_device(sc)
    b = S.Batch(ctx, [subset_struct(dev, int(off[k]), int(off[k + 1]), 0)
                      for k in range(len(off) - 1)], [cam], S.opts(), capacity)
    b.keep = dev
    return b


def _forward(b):
    from paper_2606_18588_gb300 import splx as S
    rgb = torch.empty(b.rgb_off[-1], device="cuda")
    b.forward(rgb)
    torch.cuda.synchronize()
    assert b.status()[0] == S.OK
    return rgb, b.counters()


@pytest.mark.parametrize("form", ["stale", "order set later", "persistent"])
def test_prefixes_stay_where_no_waves_were_counted(ctx, form):
    sc, off = _open_scene()
    b = _batch(ctx, sc, off)
    if form == "order set later":
        _forward(b)
        b.set_order(ORDER)
    else:
        b.set_order(ORDER)
        if form == "persistent":
            b.set_launch(4)
        else:
            b.set_stale([torch.full((CAM.height * CAM.width,), 255, dtype=torch.uint8,
                                    device="cuda")])
        _, c = _forward(b)
        assert c["skipped_items"] == 0 and 0 < c["prefix_items"] < 3 and c["retried_items"] == 0
    b.tune_prefix_sort()
    _, c = _forward(b)
    assert 0 < c["prefix_items"] < 3 and c["retried_items"] == 0
    b.close()


def _launches(ctx, b):
    """Kernel launches of a forward, and its images and counters."""
    n0 = ctx.launch_count
    rgb, c = _forward(b)
    return ctx.launch_count - n0, rgb, c


def test_one_launch_lasts_as_long_as_what_it_was_found_on(ctx):
    sc, off = _open_scene(0)
    b = _batch(ctx, sc, off)
    b.set_order(ORDER)
    waves, ref, c = _launches(ctx, b)
    assert c["skipped_items"] == 0 and c["prefix_items"] == 0
    b.tune_prefix_sort()
    one, rgb, _ = _launches(ctx, b)
    assert one == waves - 5 and torch.equal(rgb, ref)  # 2 x (sort, forward, retries' two) - 3
    b.tune_prefix_sort()  # the counts of a forward in one launch say the same
    assert _launches(ctx, b)[0] == one
    # persistent CTAs and a stale state go their own way, and it is there again after them
    b.set_launch(4)
    n, rgb, _ = _launches(ctx, b)
    assert n == waves and torch.equal(rgb, ref)
    b.set_launch(0)
    assert _launches(ctx, b)[0] == one
    for change in (lambda: b.set_cameras([CAM]), lambda: b.set_order(ORDER),
                   lambda: b.set_prefix_sort(True)):
        change()
        n, rgb, _ = _launches(ctx, b)
        assert n == waves and torch.equal(rgb, ref)
        b.tune_prefix_sort()
        assert _launches(ctx, b)[0] == one
    b.close()


def _walled_scene(x0, x1, n=3_000):
    """Two opaque walls, one behind the other, between x0 and x1 (two subsets: one alone leaves
    eps_T), and faint Gaussians everywhere behind them (the third)."""
    rng = np.random.default_rng(3)
    parts = []
    for z in (-1.3, -1.15):
        m = np.stack([rng.uniform(x0, x1, n), rng.uniform(-0.8, 0.8, n),
                      rng.uniform(z, z + 0.1, n)], 1).astype(np.float32)
        parts.append(I.Scene(m, np.full((n, 3), -2.6, np.float32),
                             np.tile(np.float32([1, 0, 0, 0]), (n, 1)),
                             np.full(n, 4.0, np.float32), np.zeros((n, 1, 3), np.float32), 0))
    faint = I.uniform_scene(900_000, 61, 0, log_scale_mu=-2.6, extent=1.0)
    faint.means[:, 0] *= 2.4
    faint.opacity_logits[:] = -4.5
    parts.append(faint)
    sc = I.Scene(*[np.concatenate(a) for a in zip(*[p.arrays() for p in parts])], 0)
    return sc, np.array([0, n, 2 * n, 2 * n + 900_000])


WALL_ORDER = np.array([[0, 1, 2]])


def test_one_launch_is_weighed_again(ctx):
    # found on a view that looks past the walls (and hands its prefixes back: whole sorts from
    # then on); then the camera moves before them: a forward in waves skips, and stays in waves
    sc, off = _walled_scene(1.4, 2.6)
    cam = I.pinhole(256, 192, 40.0, (-0.8, 0.0, -3.0), (-0.8, 0.0, 0.0))
    b = _batch(ctx, sc, off, cam, 1 << 23)
    b.set_order(WALL_ORDER)
    waves, _, c = _launches(ctx, b)
    assert c["skipped_items"] == 0 and 4 * c["retried_items"] > c["prefix_items"] > 0
    b.tune_prefix_sort()
    waves -= 3  # (no second forward)
    assert _launches(ctx, b)[0] == waves - 6  # 3 x (sort, long sort, forward) - 3
    b.set_cameras([I.pinhole(256, 192, 30.0, (2.0, 0.0, -3.0), (2.0, 0.0, 0.0))])
    n, ref, c = _launches(ctx, b)
    assert n == waves and 4 * c["skipped_items"] > 192
    b.tune_prefix_sort()
    n, rgb, _ = _launches(ctx, b)
    assert n == waves and torch.equal(rgb, ref)
    b.close()


def _wall(rng, n, x, y, z, ls):
    m = np.stack([rng.uniform(*x, n), rng.uniform(*y, n), rng.uniform(z, z + 0.1, n)], 1)
    return I.Scene(m.astype(np.float32), np.full((n, 3), ls, np.float32),
                   np.tile(np.float32([1, 0, 0, 0]), (n, 1)), np.full(n, 4.0, np.float32),
                   np.zeros((n, 1, 3), np.float32), 0)


@pytest.mark.parametrize("form", ["handed back", "few items"])
def test_waves_stay_where_skipping_saves_most_keys(ctx, form):
    """Two walls and what they hide.  "handed back": faint Gaussians everywhere, whose lists
    outlast their prefixes beside the walls, where most of them are, behind them.  "few
    items": a clump behind a small part of walls that fill the view, so that few items are
    skipped, with most of the keys."""
    rng = np.random.default_rng(8)
    if form == "handed back":
        cam = I.pinhole(256, 192, 60.0, (0.0, 0.0, -3.0), (0.0, 0.0, 0.0))
        walls = [_wall(rng, 4_000, (-0.5, 1.3), (-0.9, 0.9), z, -2.8) for z in (-1.3, -1.15)]
        back = I.uniform_scene(400_000, 5, 0, log_scale_mu=-2.6, extent=1.0)
        back.means[:, :2] *= 1.7
        back.opacity_logits[:] = -4.0
    else:
        cam = I.pinhole(512, 384, 60.0, (0.0, 0.0, -3.0), (0.0, 0.0, 0.0))
        walls = [_wall(rng, 9_000, (-1.3, 1.3), (-1.0, 1.0), z, -2.8) for z in (-1.3, -1.15)]
        back = I.uniform_scene(40_000, 5, 0, log_scale_mu=-2.5, log_scale_sigma=0.1, extent=0.05)
    parts = [*walls, back]
    sc = I.Scene(*[np.concatenate(a) for a in zip(*[p.arrays() for p in parts])], 0)
    b = _batch(ctx, sc, np.cumsum([0] + [p.n for p in parts]), cam, 1 << 23)
    b.set_order(WALL_ORDER)
    waves, ref, c = _launches(ctx, b)
    inside = 3 * ((cam.width + 15) // 16) * ((cam.height + 15) // 16) - c["outside_items"]
    if form == "handed back":
        assert 4 * c["retried_items"] > c["prefix_items"] > 0
    else:
        assert 0 < 16 * c["skipped_items"] < inside and c["prefix_items"] == 0
    b.tune_prefix_sort()
    n, rgb, c = _launches(ctx, b)
    assert n == (waves - 3 if form == "handed back" else waves) and torch.equal(rgb, ref)
    assert c["prefix_items"] == 0  # (off where they were handed back)
    b.close()
