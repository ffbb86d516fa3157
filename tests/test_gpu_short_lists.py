"""The backward rasteriser's walk of short lists (at most 32 entries: from the list's end, not
from the last contributor) and of longer ones, side by side with empty tiles: lists of 31, 32
and 33 entries, pixels that stop inside them or have no adjoint (half of every tile, whole
tiles), in small and in larger launches, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_18588_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
GROUPS = ("means", "log_scales", "quats", "opacity_logits", "sh")


@pytest.fixture(scope="module")
def ctx():
    from paper_2606_18588_gb300 import splx as S
    c = S.Context()
    yield c
    c.close()


def _scene(n, opaque):
    rng = np.random.default_rng(500 + n)
    m = rng.uniform(-0.25, 0.25, (n, 3)).astype(np.float32)
    return I.Scene(m, rng.uniform(-3.2, -1.8, (n, 3)).astype(np.float32),
                   rng.standard_normal((n, 4)).astype(np.float32),
                   rng.normal(3.0 if opaque else -2.0, 1.0, n).astype(np.float32),
                   rng.uniform(-1.0, 1.5, (n, 1, 3)).astype(np.float32), 0)


@pytest.mark.parametrize("opaque", [False, True])
@pytest.mark.parametrize("n", [31, 32, 33])
@pytest.mark.parametrize("size", [(61, 45), (528, 512)])  # 12 and 1056 tiles of 16 x 16
def test_short_lists(ctx, size, n, opaque):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import GRAD_TOL, backward_view, band_share, rel_l2, render_view, to_device
    sc = _scene(n, opaque)
    off = np.array([0, n])
    cam = I.pinhole(*size, 60.0, (0.0, 0.0, -2.0), (0.0, 0.0, 0.0))
    ref = O.render_view(sc, off, cam, O.opts(), bounds=True)
    band_share(ref["amb"], budget=0.02, label=f"{size} n {n}")
    rng = np.random.default_rng(n)
    dl = rng.standard_normal((3, cam.height, cam.width)) * (ref["amb"] == 0)
    dl[:, (np.arange(cam.height) // 4) % 2 == 1] = 0.0  # half of every tile's rows
    dl[:, :, cam.width // 2:cam.width // 2 + 40] = 0.0  # whole tiles
    gref = O.backward_view(sc, off, cam, dl, None, O.opts())
    dev = to_device(sc)
    for tile in (8, 16, 32):
        o = S.opts(tile=tile)
        _, _, parts, states = render_view(ctx, dev, off, cam, o, 0)
        longest = max(int((r[1] - r[0])) for r in states[0].export()[0])
        assert longest == n if tile == 32 and size[0] < 100 else longest <= n
        g = backward_view(ctx, dev, off, cam, o, 0, parts, states,
                          torch.from_numpy(dl.astype(np.float32)).cuda())
        for k, gr in zip(GROUPS, gref):
            e = rel_l2(g[k].cpu().numpy(), gr)
            assert e <= GRAD_TOL, (tile, k, e)
        for st in states:
            st.close()
