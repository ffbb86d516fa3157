"""The structural loss at the edges of its 32x32 tiles: images of one pixel, one short of, at
and one past a tile side, thinner than the window, and flat ones (variances zero)."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("W,H", [(1, 1), (31, 33), (32, 32), (33, 31), (37, 4), (3, 70), (65, 97)])
@pytest.mark.parametrize("flat", [False, True])
def test_loss_at_tile_edges(W, H, flat):
    from paper_2606_18588_gb300 import splx as S
    ctx = S.Context()
    rng = np.random.default_rng(W * 100 + H)
    x = (np.full((3, H, W), 0.4) if flat else rng.uniform(0, 1, (3, H, W))).astype(np.float32)
    y = (np.full((3, H, W), 0.7) if flat
         else np.clip(x + rng.normal(0, 0.1, x.shape), 0, 1)).astype(np.float32)
    loss = torch.zeros(1, device="cuda")
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    dL = torch.empty_like(xd)
    S.loss_l1_dssim(ctx, xd, yd, loss, dL, 0.2)
    torch.cuda.synchronize()
    got, g = float(loss.item()), dL.cpu().numpy()
    ctx.close()
    ref, rg = O.loss_l1_dssim([x], [y], 0.2)
    assert abs(got - ref) <= 1e-5 * abs(ref) + 1e-7
    assert np.abs(g - rg[0]).max() <= 1e-4 * np.abs(rg[0]).max()
