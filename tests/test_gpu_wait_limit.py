"""A bounded device wait that runs out (the long-segment sort's, whose limit a caller can set to
nothing) is reported on every path: a server's requests fail with it, per-view, allocation-free
and batched renders show it in the status; with the limit restored the same objects render
what they should."""
import numpy as np
import pytest

from paper_2606_18588_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture()
def ctx():
    from paper_2606_18588_gb300 import splx as S
    c = S.Context()
    yield c
    c.close()


def _scene():
    # 60k Gaussians over a few tiles: lists of several chunks of 4096 keys, merged in rounds
    sc = I.uniform_scene(60_000, 91, 0, log_scale_mu=-3.0, extent=0.3)
    sc.opacity_logits[:] = -4.0
    return sc


CAM = I.pinhole(64, 48, 60.0, (0.0, 0.0, -3.0), (0.0, 0.0, 0.0))


def _serve(srv, cam):
    out = torch.full((3, cam.height, cam.width), float("nan"), device="cuda")
    rid = srv.submit(cam, out)
    done = {}
    while rid not in done:
        done.update(srv.poll())
    torch.cuda.synchronize()
    return out, done[rid]


def test_server_requests_fail_with_the_timeout(ctx):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import subset_struct, to_device
    sc = _scene()
    dev = to_device(sc)
    srv = S.Server(ctx, [subset_struct(dev, 0, sc.n, 0)], S.opts(), 1 << 30, slots=2, max_views=2)
    ref, st = _serve(srv, CAM)
    assert st == S.OK
    ctx.set_wait_limit(0)
    _, st = _serve(srv, CAM)
    assert st == S.ERR_TIMEOUT
    assert ctx.device_status() == S.ERR_TIMEOUT and ctx.device_status() == S.OK
    # a launch without long lists has nothing to wait for
    far = I.pinhole(64, 48, 60.0, (0.0, 0.0, 3.0), (0.0, 0.0, 6.0))
    assert _serve(srv, far)[1] == S.OK
    ctx.set_wait_limit(1 << 20)
    out, st = _serve(srv, CAM)
    assert st == S.OK and torch.equal(out, ref)
    assert ctx.device_status() == S.OK
    srv.close()


def test_renders_report_the_timeout(ctx):
    from paper_2606_18588_gb300 import splx as S
    from gpu_util import subset_struct, to_device
    sc = _scene()
    dev = to_device(sc)
    sub = subset_struct(dev, 0, sc.n, 0)
    part = S.new_partial(CAM.height, CAM.width)
    b = S.Batch(ctx, [sub], [CAM], S.opts())
    b.set_prefix_sort(False)
    rgb = torch.empty(b.rgb_off[-1], device="cuda")
    ref = None
    for polls, want in ((1 << 20, S.OK), (0, S.ERR_TIMEOUT), (1 << 20, S.OK)):
        ctx.set_wait_limit(polls)
        S.render_partial(ctx, sub, CAM, S.opts(), part, keep_state=False)
        assert ctx.device_status() == want
        b.forward(rgb)
        assert b.status()[0] == want
        assert ctx.device_status() == want
        if want == S.OK:
            got = torch.cat([part["rgb"].reshape(-1), rgb])
            ref = got.clone() if ref is None else ref
            assert torch.equal(got, ref)
    for bad in (-1, (1 << 20) + 1):
        with pytest.raises(S.SplxError):
            ctx.set_wait_limit(bad)
    b.close()
