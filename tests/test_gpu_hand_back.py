"""Tiles whose nearest depth bin alone holds more keys than a selected prefix may (every key of
the subset at one depth): the forward hands them to the whole sort without walking, in the
first and in later saturation-skipping waves, with one CTA per item and with persistent CTAs,
and forward after forward equals whole sorts bit for bit (a warp that took the unsorted list, or
an item counted twice in the prefix transmittance, would show in the images)."""
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


def _sheets():
    # three sheets of faint Gaussians facing the camera, each at one depth (one subset each):
    # no list longer than a prefix has one, and no pixel saturates before the last sheet
    parts = []
    for i, z in enumerate((-0.6, 0.0, 0.6)):
        s = I.uniform_scene(8_000, 80 + i, 0, log_scale_mu=-3.0, extent=0.25)
        s.means[:, 2] = z
        s.opacity_logits[:] = -4.8 + 0.3 * s.opacity_logits
        parts.append(s)
    return parts


@pytest.mark.parametrize("persist", [0, 1])
@pytest.mark.parametrize("waves", [True, False])
@pytest.mark.parametrize("tile", [8, 16, 32])
def test_lists_without_a_prefix(ctx, tile, waves, persist):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import subset_struct, to_device
    parts = _sheets()
    sc = I.Scene(*[np.concatenate(a) for a in zip(*[p.arrays() for p in parts])], 0)
    off = np.cumsum([0] + [p.n for p in parts])
    cams = [I.pinhole(64, 64, 60.0, (0.0, 0.0, -3.0), (0, 0, 0)),
            I.pinhole(75, 50, 60.0, (0.0, 0.0, -3.0), (0, 0, 0))]
    dev = to_device(sc)
    subs = [subset_struct(dev, int(off[k]), int(off[k + 1]), 0) for k in range(3)]
    b = S.Batch(ctx, subs, cams, S.opts(tile=tile))
    if waves:
        b.set_order(np.array([[0, 1, 2], [0, 1, 2]]))
    out = []
    for prefix in (False, True):
        b.set_prefix_sort(prefix)
        b.set_launch(persist if prefix else 0)
        for rep in range(20 if prefix else 1):
            rgb = torch.empty(b.rgb_off[-1], device="cuda")
            T = torch.empty(b.total_pixels, device="cuda")
            b.forward(rgb, T)
            out.append((rgb, T))
        torch.cuda.synchronize()
        assert b.status()[0] == S.OK
    c = b.counters()
    # every list beyond a prefix's 2048 keys went that way, in each wave
    want = sum(int((np.diff(O.tile_lists(p, cam, tile)[0]) > 2048).sum())
               for p in parts for cam in cams)
    assert c["retried_items"] == want >= 8 and c["prefix_items"] == 0
    for rgb, T in out[1:]:
        assert torch.equal(rgb, out[0][0]) and torch.equal(T, out[0][1])
    b.close()
