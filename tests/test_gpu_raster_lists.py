"""The rasterisers at the sizes where their tile walks change shape: lists of one entry, of
odd length, around a group of 32, a half and a whole ring of 64, a staged batch of 128 and
beyond; images ragged against every tile side; pixels that stop inside a list and pixels
that never do; a threshold of zero (every entry of a rectangle is taken); a colour that is
not finite.  Forward and gradients against the oracle, forward bit-identical across tiles."""
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
    """n Gaussians in front of the middle of the view, from needles to blobs."""
    rng = np.random.default_rng(1000 + n)
    m = rng.uniform(-0.4, 0.4, (n, 3)).astype(np.float32)
    ls = rng.uniform(-4.5, -1.6, (n, 3)).astype(np.float32)
    q = rng.standard_normal((n, 4)).astype(np.float32)
    logit = rng.normal(2.0 if opaque else -2.5, 1.0, n).astype(np.float32)
    sh = rng.uniform(-1.0, 1.5, (n, 1, 3)).astype(np.float32)
    return I.Scene(m, ls, q / np.linalg.norm(q, axis=1, keepdims=True), logit, sh, 0)


CAM = I.pinhole(43, 27, 60.0, (0.0, 0.0, -2.0), (0.0, 0.0, 0.0))


@pytest.mark.parametrize("opaque", [False, True])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 65, 127, 129, 300])
def test_lists_of_every_length(ctx, n, opaque):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import (GRAD_TOL, PIXEL_TOL, backward_view, band_share, check_band, rel_l2,
                          render_view, to_device)
    sc = _scene(n, opaque)
    off = np.array([0, n])
    dev = to_device(sc)
    amin = 0.0 if n == 33 else 1.0 / 255.0
    ref = O.render_view(sc, off, CAM, O.opts(alpha_min=amin), bounds=True)
    fb, amb = ref["flip"], ref["amb"]
    # (the band grows with the alphas a pixel evaluates: 2.4e-5 each and 1e-3 a stop)
    budget = 0.02
    rng = np.random.default_rng(7)
    dl = rng.standard_normal((3, CAM.height, CAM.width)) * (amb == 0)
    gref = O.backward_view(sc, off, CAM, dl, None, O.opts(alpha_min=amin))
    first = None
    for tile in (8, 16, 32):
        o = S.opts(tile=tile, alpha_min=amin)
        img, T, parts, states = render_view(ctx, dev, off, CAM, o, 0)
        got = {k: v.cpu().numpy() for k, v in parts[0].items()}
        check_band(got["rgb"], ref["Cp"][0], amb, fb["partC"][0], budget=budget, label="C")
        check_band(got["T"], ref["Tp"][0], amb, fb["partT"][0], budget=budget, label="T")
        if first is None:
            first = got
        for k in ("rgb", "T", "depth"):
            assert np.array_equal(got[k], first[k]), (tile, k)
        band_share(amb, budget=budget, label=f"n {n} tile {tile} gradients")
        g = backward_view(ctx, dev, off, CAM, o, 0, parts, states,
                          torch.from_numpy(dl.astype(np.float32)).cuda())
        for k, gr in zip(GROUPS, gref):
            e = rel_l2(g[k].cpu().numpy(), gr)
            assert e <= GRAD_TOL, (tile, k, e)
        for st in states:
            st.close()
    assert np.abs(got["T"] - ref["Tp"][0])[amb == 0].max(initial=0.0) <= PIXEL_TOL


@pytest.mark.parametrize("tile", [8, 16, 32])
def test_infinite_colour_stays_in_its_pixels(ctx, tile):
    """A colour that overflows shows only where its Gaussian is blended, in the image and in
    the gradients; everything else is as if it had any other colour."""
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import backward_view, render_view, to_device
    n, bad = 200, 117
    sc = _scene(n, False)
    sc.log_scales[bad] = -4.0  # a small footprint
    off = np.array([0, n])
    o = S.opts(tile=tile)
    outs = []
    for colour in (1.0, np.inf):
        sc.sh[bad] = colour
        dev = to_device(sc)
        img, T, parts, states = render_view(ctx, dev, off, CAM, o, 0)
        dl = torch.ones_like(img)
        g = backward_view(ctx, dev, off, CAM, o, 0, parts, states, dl)
        outs.append((parts[0]["rgb"].cpu().numpy(), parts[0]["T"].cpu().numpy(),
                     g["sh"].cpu().numpy(), g["opacity_logits"].cpu().numpy()))
        for st in states:
            st.close()
    (c0, t0, s0, _), (c1, t1, s1, l1) = outs
    assert np.array_equal(t0, t1)
    hit = ~np.isfinite(c1).all(axis=0)
    assert 0 < hit.sum() < 100
    assert np.array_equal(c0[:, ~hit], c1[:, ~hit])
    # a Gaussian that shares no pixel with it has finite gradients
    alone = np.isfinite(l1)
    assert 0 < alone.sum() < n
    fin = np.isfinite(s1).all(axis=(1, 2))
    assert np.allclose(s0[fin], s1[fin], rtol=1e-4, atol=1e-6)


@pytest.mark.parametrize("w", [512, 528])
def test_backward_on_both_sides_of_its_launch_rule(ctx, w):
    """1024 and 1056 tiles of 16x16 (the backward's forms for small and for larger launches)
    against the 8x8 tiles' backward and the oracle: the same sums, added in another order."""
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import GRAD_TOL, backward_view, band_share, rel_l2, render_view, to_device
    n = 400
    sc = _scene(n, False)
    off = np.array([0, n])
    cam = I.pinhole(w, 512, 60.0, (0.0, 0.0, -2.0), (0.0, 0.0, 0.0))
    dev = to_device(sc)
    ref = O.render_view(sc, off, cam, O.opts(), bounds=True)
    rng = np.random.default_rng(9)
    dl = rng.standard_normal((3, 512, w)) * (ref["amb"] == 0)
    band_share(ref["amb"], budget=0.02, label=f"{w} x 512")
    gref = O.backward_view(sc, off, cam, dl, None, O.opts())
    got = {}
    for tile in (16, 8):
        o = S.opts(tile=tile)
        _, _, parts, states = render_view(ctx, dev, off, cam, o, 0)
        got[tile] = backward_view(ctx, dev, off, cam, o, 0, parts, states,
                                  torch.from_numpy(dl.astype(np.float32)).cuda())
        for st in states:
            st.close()
    for k, gr in zip(GROUPS, gref):
        a, b = got[16][k].cpu().numpy(), got[8][k].cpu().numpy()
        assert rel_l2(a, gr) <= GRAD_TOL, k
        assert rel_l2(a, b) <= 1e-5, k
