"""Composition and its adjoint with and without visible regions: patches of a tile, or 32
consecutive pixels of a view (whose last warp is not full), one subset, and more subsets than
registers hold.  Subsets outside a tile are empty there, so both give the same bit for bit."""
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


@pytest.mark.parametrize("K", [1, 2, 3, 8, 16, 17, 32, 33, 64])
@pytest.mark.parametrize("tile", [8, 16, 32])
def test_regions_do_not_change_the_composition(ctx, K, tile):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import params_struct, rel_l2, subset_struct, to_device, zeros_like_params
    n = 40 * K
    sc = I.uniform_scene(n, 300 + K, 0, log_scale_mu=-2.0)
    sc = sc.take(np.argsort(sc.means[:, 0], kind="stable"))  # slabs, each seen in part of a view
    off = np.linspace(0, n, K + 1).astype(np.int64)
    # 1419, 31 and 2880 pixels: no multiple of a warp's 32 but the last
    cams = [I.pinhole(w, h, 70.0, (0.0, 0.0, -2.5), (0.0, 0.0, 0.0))
            for w, h in ((43, 33), (31, 1), (64, 45))]
    dev = to_device(sc)
    b = S.Batch(ctx, [subset_struct(dev, int(off[k]), int(off[k + 1]), 0) for k in range(K)],
                cams, S.opts(tile=tile, bg=(0.3, 0.2, 0.1)))
    rng = np.random.default_rng(K)
    dC = torch.from_numpy(rng.standard_normal(b.rgb_off[-1]).astype(np.float32)).cuda()
    dT = torch.from_numpy(rng.standard_normal(b.total_pixels).astype(np.float32)).cuda()
    out = []
    for regions in (True, False):
        b.set_visibility(regions)
        rgb = torch.full((b.rgb_off[-1],), float("nan"), device="cuda")
        T = torch.full((b.total_pixels,), float("nan"), device="cuda")
        g = zeros_like_params(dev)
        b.forward(rgb, T)
        b.backward(dC, dT, [params_struct(g, int(off[k]), int(off[k + 1]), 0) for k in range(K)])
        torch.cuda.synchronize()
        out.append((rgb, T, g))
    b.close()
    (c0, t0, g0), (c1, t1, g1) = out
    assert torch.equal(c0, c1) and torch.equal(t0, t1)
    assert torch.isfinite(c0).all() and (t0 < 0.9).any()
    for k in g0:
        assert rel_l2(g1[k].cpu().numpy(), g0[k].cpu().numpy()) <= 1e-5, k
