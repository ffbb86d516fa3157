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


def _batch(ctx, sc, off, cam=CAM):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import subset_struct, to_device
    dev = to_device(sc)
    b = S.Batch(ctx, [subset_struct(dev, int(off[k]), int(off[k + 1]), 0)
                      for k in range(len(off) - 1)], [cam], S.opts(), 1 << 20)
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
    faint = I.uniform_scene(2_000, 61, 0, log_scale_mu=-3.0, extent=1.0)
    faint.means[:, 0] *= 2.4
    faint.opacity_logits[:] = -3.0
    parts.append(faint)
    sc = I.Scene(*[np.concatenate(a) for a in zip(*[p.arrays() for p in parts])], 0)
    return sc, np.array([0, n, 2 * n, 2 * n + 2_000])


WALL_ORDER = np.array([[0, 1, 2]])


def test_one_launch_is_weighed_again(ctx):
    # found on a view that looks past the walls; then the camera moves before them: a forward
    # in waves skips, and stays in waves
    sc, off = _walled_scene(1.4, 2.6)
    b = _batch(ctx, sc, off, I.pinhole(256, 192, 40.0, (-0.8, 0.0, -3.0), (-0.8, 0.0, 0.0)))
    b.set_order(WALL_ORDER)
    waves, _, c = _launches(ctx, b)
    assert c["skipped_items"] == 0
    b.tune_prefix_sort()
    one = _launches(ctx, b)[0]
    assert one < waves
    b.set_cameras([I.pinhole(256, 192, 30.0, (2.0, 0.0, -3.0), (2.0, 0.0, 0.0))])
    n, ref, c = _launches(ctx, b)
    assert n == waves and 4 * c["skipped_items"] > 192
    b.tune_prefix_sort()
    n, rgb, _ = _launches(ctx, b)
    assert n == waves and torch.equal(rgb, ref)
    b.close()
