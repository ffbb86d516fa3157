"""What splx_batch_tune_prefix_sort decides: a stale saturation state, an eager forward made
before the subset orders were set and persistent CTAs leave the selected prefixes on (there are
no waves to replace, or none were counted)."""
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
                      for k in range(len(off) - 1)], [cam], S.opts())
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
