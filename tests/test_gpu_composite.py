"""Composition and its adjoint over every number of subsets that changes their form (four,
eight and sixteen in registers, more through arrays, more than 32 pointers per warp), on
images ragged against the tiles whose patches the warps take: against the oracle, and the
batch (which leaves out subsets whose visible region misses a tile) against the per-view
path."""
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


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("K", [1, 4, 5, 8, 9, 16, 17, 33, 64])
def test_composition_of_k_subsets(ctx, K, tile):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import (GRAD_TOL, PIXEL_TOL, backward_view, band_share, check_band,
                          params_struct, rel_l2, render_view, subset_struct, to_device,
                          zeros_like_params)
    n = 12 * K + 5
    sc = I.uniform_scene(n, 900 + K, 1, log_scale_mu=-2.2)
    sc.opacity_logits[:] = sc.opacity_logits - 1.0
    # depth slabs, so that the subsets' order is that of their depths; some are empty
    sc = sc.take(np.argsort(sc.means[:, 2], kind="stable"))
    off = np.linspace(0, n, K + 1).astype(np.int64)
    if K > 4:
        off[3] = off[2]
    cam = I.pinhole(45, 29, 60.0, (0.0, 0.0, -3.0), (0.0, 0.0, 0.0))
    dev = to_device(sc)
    o = S.opts(tile=tile, bg=(0.2, 0.1, 0.3))
    oo = O.opts(bg=(0.2, 0.1, 0.3))
    ref = O.render_view(sc, off, cam, oo, bounds=True)
    fb, amb = ref["flip"], ref["amb"]
    budget = 0.03  # (K keys and cuts per pixel beside the alphas)
    img, T, parts, states = render_view(ctx, dev, off, cam, o, 1)
    check_band(img.cpu().numpy(), ref["image"], amb, fb["image"], budget=budget, label="image")
    check_band(T.cpu().numpy(), ref["T"], amb, fb["T"], tol=PIXEL_TOL, budget=budget, label="T")
    rng = np.random.default_rng(K)
    dl = rng.standard_normal((3, cam.height, cam.width)) * (amb == 0)
    dT = rng.standard_normal((cam.height, cam.width)) * (amb == 0)
    band_share(amb, budget=budget, label=f"K {K} gradients")
    dl_d = torch.from_numpy(dl.astype(np.float32)).cuda()
    dT_d = torch.from_numpy(dT.astype(np.float32)).cuda()
    g = backward_view(ctx, dev, off, cam, o, 1, parts, states, dl_d, dT_d)
    for k, gr in zip(GROUPS, O.backward_view(sc, off, cam, dl, dT, oo)):
        assert rel_l2(g[k].cpu().numpy(), gr) <= GRAD_TOL, k
    for st in states:
        st.close()
    b = S.Batch(ctx, [subset_struct(dev, int(off[k]), int(off[k + 1]), 1) for k in range(K)], [cam], o)
    rgb = torch.empty(b.rgb_off[-1], device="cuda")
    Tb = torch.empty(b.total_pixels, device="cuda")
    b.forward(rgb, Tb)
    gb = zeros_like_params(dev)
    b.backward(dl_d.reshape(-1), dT_d.reshape(-1),
               [params_struct(gb, int(off[k]), int(off[k + 1]), 1) for k in range(K)])
    torch.cuda.synchronize()
    same = torch.equal(b.views(rgb)[0], img) and torch.equal(Tb.view_as(T), T)
    b.close()
    assert same
    for k in GROUPS:
        assert rel_l2(gb[k].cpu().numpy(), g[k].cpu().numpy()) <= 1e-5, k
