"""The projection's two forms (coefficients staged once for batches of many views, read per
view for few) on subsets that begin and end inside a warp, counts that are no multiple of 32,
coefficients that are not 16-byte aligned, and every SH degree: a batch of nine views equals
the views rendered one by one, bit for bit."""
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


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("deg", [0, 1, 2, 3])
def test_many_views_equal_single_views(ctx, deg, shift):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import subset_struct, to_device
    n = 1501
    rng = np.random.default_rng(deg)
    m = rng.uniform(-1.5, 1.5, (n, 3)).astype(np.float32)
    q = rng.standard_normal((n, 4)).astype(np.float32)
    sc = I.Scene(m, rng.uniform(-4.5, -2.0, (n, 3)).astype(np.float32), q,
                 rng.normal(0.0, 1.5, n).astype(np.float32),
                 rng.normal(0.0, 0.4, (n, (deg + 1) ** 2, 3)).astype(np.float32), deg)
    off = [0, 7, 71, 640, 641, n]
    a = np.linspace(0.0, 5.0, 9)
    cams = [I.pinhole(83, 61, 70.0, (3.0 * np.sin(t), 0.4 * t - 1.0, 3.0 * np.cos(t)), (0, 0, 0))
            for t in a]
    dev = to_device(sc)
    room = torch.empty(dev["sh"].numel() + 4, device="cuda")
    sh = room[shift:shift + dev["sh"].numel()].view_as(dev["sh"])
    sh.copy_(dev["sh"])
    dev["sh"] = sh
    subs = [subset_struct(dev, off[k], off[k + 1], deg) for k in range(len(off) - 1)]

    def render(cs):
        b = S.Batch(ctx, subs, cs, S.opts())
        rgb = torch.empty(b.rgb_off[-1], device="cuda")
        b.forward(rgb)
        out = [v.clone() for v in b.views(rgb)]
        torch.cuda.synchronize()
        b.close()
        return out

    many = render(cams)
    assert float(many[0].abs().sum()) > 0.0
    for v, cam in enumerate(cams):
        assert torch.equal(many[v], render([cam])[0]), v
