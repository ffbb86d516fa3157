"""The loss's sums keep at least the 53 bits of a double: one channel's |x - y| holds 3, 3 x 2^-24
and 3 x 2^-51 and zeros elsewhere, so that the mean lies just above the middle of two FP32
numbers, and only the smallest term, 2^-51 of the sum, says which is nearer."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("where", [((0, 0), (1, 0), (2, 0)),        # one thread's pixels
                                   ((0, 0), (0, 1), (0, 17)),       # one warp's
                                   ((0, 3), (9, 9), (31, 31)),      # one tile's
                                   ((31, 31), (0, 0), (30, 2))])
@pytest.mark.parametrize("entry", ["image", "batch"])
def test_smallest_term_decides_the_rounding(where, entry):
    from paper_2606_18588_gb300 import splx as S
    terms = (3.0, 3.0 * 2.0 ** -24, 3.0 * 2.0 ** -51)
    x = np.zeros((3, 32, 32), np.float32)
    for (r, c), t in zip(where, terms):
        x[1, r, c] = t
    exact = sum(terms) / x.size  # in doubles: 2^-10 (1 + 2^-24 + 2^-51), then to FP32
    want = np.float32(exact)
    assert want == np.float32(2.0 ** -10 * (1.0 + 2.0 ** -23))
    assert np.float32((terms[0] + terms[1]) / x.size) == np.float32(2.0 ** -10)
    ctx = S.Context()
    loss = torch.zeros(1, device="cuda")
    xd, yd = torch.from_numpy(x).cuda(), torch.zeros(3, 32, 32, device="cuda")
    dL = torch.empty_like(xd)
    if entry == "image":
        S.loss_l1_dssim(ctx, xd, yd, loss, dL, 0.0)
    else:
        from gpu_util import subset_struct, to_device
        from paper_2606_18588_gb300 import inputs as I
        dev = to_device(I.uniform_scene(10, 1))
        cam = I.pinhole(32, 32, 60.0, (0.0, 0.0, -3.0), (0.0, 0.0, 0.0))
        b = S.Batch(ctx, [subset_struct(dev, 0, 10, 0)], [cam], S.opts())
        b.loss_l1_dssim(xd.reshape(-1), yd.reshape(-1), loss, dL.reshape(-1), 0.0)
        torch.cuda.synchronize()
        b.close()
    torch.cuda.synchronize()
    assert np.float32(loss.item()) == want
    ctx.close()
