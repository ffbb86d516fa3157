"""What users of the framework have it do, as measurable cases.

Each case is one call (or the few calls of one pass) through the public entry points:
training steps over batches of views, the autograd renderer, per-view local renders with
and without a forward state, forward-only batches, the render server, and the single
stages that a program also calls by themselves (composition, the photometric loss, Adam).
Scenes, cameras and targets follow paper_2606_18588_gb300/inputs.py, drawn on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_18588_gb300 import inputs as I
from paper_2606_18588_gb300 import serve
from paper_2606_18588_gb300 import splx as S
from paper_2606_18588_gb300.train import DEFAULT_LR, GROUPS, BatchedStep, Renderer
from paper_2606_18588_gb300.visibility import front_to_back, orders_for_views

RESOLUTIONS = ((512, 512), (1280, 720), (1920, 1080), (3840, 2160))  # what a server is asked for


def listed():
    return [
        # the smallest render: 10k Gaussians, one subset, 256 x 256, forward only
        {"name": "partial_10k_256", "kind": "partial", "scene": "uniform", "n": 10_000, "deg": 0,
         "w": 256, "h": 256, "tile": 16},
        # a latency-critical loop that cannot allocate: 50k Gaussians of SH degree 3, VGA
        {"name": "noalloc_50k_vga", "kind": "noalloc", "scene": "uniform", "n": 50_000, "deg": 3,
         "w": 640, "h": 480, "tile": 16},
        # the smallest differentiable pass: two small ragged views, loss.backward() in torch
        {"name": "autograd_12k_k2", "kind": "autograd", "scene": "cluster", "n": 12_000, "deg": 2,
         "K": 2, "views": 2, "w": 211, "h": 157, "tile": 16},
        # one full-HD view at a time: K local renders, composite, L1, backward
        {"name": "view_1m_k4_1080p", "kind": "view", "scene": "cluster", "n": 1_000_000, "deg": 3,
         "K": 4, "w": 1920, "h": 1080, "tile": 16},
        # the headline training step: 10M Gaussians, 16 views of two resolutions, captured
        {"name": "train_10m_k8_16v", "kind": "train", "scene": "cluster", "n": 10_000_000, "deg": 3,
         "K": 8, "views": 16, "w": 1600, "h": 1064, "w2": 1280, "h2": 720, "tile": 16,
         "skip": "waves", "dssim": 0.0},
        # an ordinary training step of an object-sized scene with the structural loss
        {"name": "train_600k_k4_dssim", "kind": "train", "scene": "cluster", "n": 600_000, "deg": 3,
         "K": 4, "views": 4, "w": 979, "h": 545, "w2": 979, "h2": 545, "tile": 16,
         "skip": "waves", "dssim": 0.2},
        # a large scene of which each step's few views see a part: new views every step
        {"name": "train_city_20m_k32", "kind": "train", "scene": "city", "n": 20_000_000, "deg": 3,
         "K": 32, "views": 4, "w": 1920, "h": 1080, "w2": 1920, "h2": 1080, "tile": 16,
         "skip": "waves", "dssim": 0.0},
        # forward only, a single 4K view of a resident scene
        {"name": "render_3m_k8_4k", "kind": "render", "scene": "cluster", "n": 3_000_000, "deg": 3,
         "K": 8, "views": 1, "w": 3840, "h": 2160, "tile": 16, "skip": "none"},
        # the render server: a burst of requests of mixed resolution
        {"name": "serve_4m_k8_burst", "kind": "serve", "scene": "cluster", "n": 4_000_000, "deg": 3,
         "K": 8, "requests": 12, "tile": 16},
        # the photometric loss with its gradient, one full-HD image
        {"name": "dssim_1080p", "kind": "dssim", "w": 1920, "h": 1080},
        # the stand-alone optimiser step
        {"name": "adam_2m", "kind": "adam", "n": 2_000_000, "deg": 3},
        # composition of partial images (Eq. 5) by itself
        {"name": "composite_k16", "kind": "composite", "K": 16, "w": 1600, "h": 1064},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("partial", "noalloc", "autograd", "view", "train", "train", "train", "render",
                       "serve", "dssim", "adam", "composite"))
    w, h = _log(rng, 200, 1920), _log(rng, 150, 1080)
    c = {"kind": kind, "scene": "cluster", "deg": rng.randint(0, 3), "tile": rng.choice((16, 16, 16, 8, 32))}
    if kind == "partial":
        return {**c, "scene": "uniform", "n": _log(rng, 5_000, 500_000), "w": w, "h": h}
    if kind == "noalloc":
        return {**c, "scene": "uniform", "tile": 16, "n": _log(rng, 5_000, 60_000), "w": _log(rng, 128, 800),
                "h": _log(rng, 128, 600)}
    if kind == "autograd":
        return {**c, "n": _log(rng, 8_000, 1_000_000), "K": rng.choice((1, 2, 4)),
                "views": rng.randint(1, 6), "w": w, "h": h}
    if kind == "view":
        return {**c, "n": _log(rng, 50_000, 2_000_000), "K": rng.choice((1, 2, 4, 8)), "w": w, "h": h}
    if kind == "train":
        city = rng.random() < 0.25
        n = _log(rng, 2_000_000, 16_000_000) if city else _log(rng, 100_000, 5_000_000)
        return {**c, "scene": "city" if city else "cluster", "deg": rng.choice((0, 1, 2, 3, 3, 3)), "n": n,
                "K": rng.choice((16, 32)) if city else rng.choice((1, 2, 4, 8)),
                "views": rng.randint(1, 8), "w": w, "h": h, "w2": _log(rng, 200, 1600), "h2": _log(rng, 150, 900),
                "skip": rng.choice(("waves", "waves", "stale", "none")), "dssim": rng.choice((0.0, 0.0, 0.2))}
    if kind == "render":
        return {**c, "n": _log(rng, 100_000, 6_000_000), "K": rng.choice((1, 4, 8, 16)),
                "views": rng.randint(1, 3), "w": _log(rng, 300, 3840), "h": _log(rng, 200, 2160),
                "skip": rng.choice(("waves", "none"))}
    if kind == "serve":
        return {**c, "deg": 3, "tile": 16, "n": _log(rng, 500_000, 5_000_000), "K": rng.choice((4, 8)),
                "requests": rng.randint(2, 14)}
    if kind == "dssim":
        return {"kind": kind, "w": _log(rng, 64, 3840), "h": _log(rng, 64, 2160)}
    if kind == "adam":
        return {"kind": kind, "n": _log(rng, 20_000, 6_000_000), "deg": c["deg"]}
    return {"kind": kind, "K": rng.randint(1, 32), "w": w, "h": h}


# ---------------------------------------------------------------- inputs on the GPU
def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _uniform(g, *shape, lo=0.0, hi=1.0):
    return torch.rand(*shape, generator=g, device="cuda") * (hi - lo) + lo


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _attributes(g, n, deg, log_scale_mu):
    """Everything but the means, as inputs.py draws it."""
    quats = _normal(g, n, 4)
    quats /= quats.norm(dim=1, keepdim=True)
    sh = _normal(g, n, I.n_sh_coeffs(deg), 3) * 0.2
    sh[:, 0] = (_uniform(g, n, 3) - 0.5) * (2.0 * math.sqrt(math.pi))
    return {"log_scales": _normal(g, n, 3) * 0.5 + log_scale_mu, "quats": quats,
            "opacity_logits": _normal(g, n), "sh": sh}


def _morton(p):
    lo, hi = p.amin(dim=0), p.amax(dim=0)
    q = ((p - lo) / (hi - lo).clamp_min(1e-12) * 1023.0).long().clamp_(0, 1023)
    code = torch.zeros(p.shape[0], dtype=torch.int64, device=p.device)
    for a in range(3):
        v = q[:, a]
        v = (v | (v << 16)) & 0x030000FF
        v = (v | (v << 8)) & 0x0300F00F
        v = (v | (v << 4)) & 0x030C30C3
        v = (v | (v << 2)) & 0x09249249
        code |= v << a
    return code


def _kd(means, K):
    """Median splits on the larger of the x / z extents, cells in Morton order."""
    cells = [(means, np.full(3, -np.inf), np.full(3, np.inf))]
    while len(cells) < K:
        nxt = []
        for p, lo, hi in cells:
            ext = (p.amax(dim=0) - p.amin(dim=0)).tolist()
            ax = 0 if ext[0] >= ext[2] else 2
            p = p[torch.argsort(p[:, ax], stable=True)]
            m = p.shape[0] // 2
            plane = 0.5 * (float(p[m - 1, ax]) + float(p[m, ax]))
            lhi, rlo = hi.copy(), lo.copy()
            lhi[ax] = rlo[ax] = plane
            nxt += [(p[:m], lo, lhi), (p[m:], rlo, hi)]
        cells = nxt
    cells = [(p[torch.argsort(_morton(p), stable=True)], lo, hi) for p, lo, hi in cells]
    offsets = np.concatenate([[0], np.cumsum([p.shape[0] for p, _, _ in cells])]).astype(np.int64)
    return torch.cat([p for p, _, _ in cells]), offsets, np.stack([np.stack([lo, hi]) for _, lo, hi in cells])


def _scene(case, seed):
    """(parameters, subset offsets, cells, city layout or None)."""
    n, K, g = case["n"], case.get("K", 1), _gen(seed)
    if case["scene"] == "uniform":
        p = _uniform(g, n, 3, lo=-1.0, hi=1.0)
        return {"means": p[torch.argsort(_morton(p), stable=True)].contiguous(),
                **_attributes(g, n, case["deg"], -3.5)}, np.array([0, n]), None, None
    if case["scene"] == "city":
        lay = I.city_layout(n, seed, K, case["deg"])
        count = torch.from_numpy(lay.count).cuda()
        rep = torch.repeat_interleave(torch.arange(count.numel(), device="cuda"), count)
        lo, hi = (torch.from_numpy(a).float().cuda() for a in (lay.lo, lay.hi))
        p = lo[rep] + _uniform(g, n, 3) * (hi - lo)[rep]
        cell = torch.from_numpy(np.ascontiguousarray(lay.cell)).cuda()[rep].long()
        p = p[torch.argsort((cell << 30) | _morton(p), stable=True)].contiguous()
        return {"means": p, **_attributes(g, n, case["deg"], lay.log_scale_mu)}, lay.offsets, lay.boxes, lay
    centres = _uniform(g, 64, 3, lo=-10.0, hi=10.0)
    sigma = _uniform(g, 64, 1, lo=0.5, hi=2.0)
    lab = torch.randint(0, 64, (n,), generator=g, device="cuda")
    p = centres[lab] + sigma[lab] * _normal(g, n, 3)
    for _ in range(64):  # points outside the cube are drawn again
        bad = torch.nonzero((p.abs() > 10.0).any(dim=1)).flatten()
        if not bad.numel():
            break
        p[bad] = centres[lab[bad]] + sigma[lab[bad]] * _normal(g, bad.numel(), 3)
    p, off, boxes = _kd(p.clamp_(-10.0, 10.0), K)
    mu = math.log(0.33 * (8000.0 / n) ** (1.0 / 3.0))
    return {"means": p.contiguous(), **_attributes(g, n, case["deg"], mu)}, off, boxes, None


def _cameras(case, seed, step=0):
    if case["scene"] == "uniform":
        rng = np.random.default_rng(seed)
        d = rng.normal(size=3)
        return [I.pinhole(case["w"], case["h"], 60.0, 3.0 * d / np.linalg.norm(d), (0.0, 0.0, 0.0))]
    sizes = [(case["w"], case["h"]), (case.get("w2", case["w"]), case.get("h2", case["h"]))]
    V = case.get("views", 1)
    if case["scene"] == "city":
        pick = I.step_views(seed, step, 500, V)
        pools = [I.aerial_cameras(seed, size=s) for s in sizes]
        return [pools[i % 2][j] for i, j in enumerate(pick)]
    return I.orbit_cameras(V, seed + 1, sizes)


def _subsets(p, off, deg, make=S.gaussians):
    return [make(*(p[k][int(off[i]):int(off[i + 1])] for k in GROUPS), deg) for i in range(len(off) - 1)]


def _pixels(case):
    V = case.get("views", 1)
    a, b = case["w"] * case["h"], case.get("w2", case["w"]) * case.get("h2", case["h"])
    return a * ((V + 1) // 2) + b * (V // 2)


# ---------------------------------------------------------------- prepare
def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def _prep_partial(case, seed):
    p, _, _, _ = _scene(case, seed)
    return {"case": case, "ctx": S.Context(), "keep": p, "sub": S.gaussians(*(p[k] for k in GROUPS), case["deg"]),
            "cam": _cameras(case, seed)[0], "opts": S.opts(tile=case["tile"]),
            "out": S.new_partial(case["h"], case["w"])}


def _prep_autograd(case, seed):
    p, off, _, _ = _scene(case, seed)
    ctx = S.Context()
    p = {k: v.requires_grad_() for k, v in p.items()}
    r = Renderer(ctx, p, off, case["deg"], _cameras(case, seed), S.opts(tile=case["tile"]))
    return {"case": case, "p": p, "r": r, "target": _uniform(_gen(seed, 1), 3 * _pixels(case))}


def _prep_view(case, seed):
    p, off, _, _ = _scene(case, seed)
    K, h, w = case["K"], case["h"], case["w"]
    g = {k: torch.zeros_like(v) for k, v in p.items()}
    return {"case": case, "ctx": S.Context(), "keep": p, "subs": _subsets(p, off, case["deg"]), "g": g,
            "grads": _subsets(g, off, case["deg"], S.params), "cam": _cameras(case, seed)[0],
            "opts": S.opts(tile=case["tile"]), "parts": [S.new_partial(h, w) for _ in range(K)],
            "img": torch.empty(3, h, w, device="cuda"), "dL": torch.empty(3, h, w, device="cuda"),
            "loss": torch.zeros(1, device="cuda"), "target": _uniform(_gen(seed, 1), 3, h, w)}


_TRAIN_STREAM = None


def _train_stream():
    """The stream of a program's training steps (a captured step cannot run on the legacy
    default stream): one for all, so that steps follow each other as in one training run."""
    global _TRAIN_STREAM
    if _TRAIN_STREAM is None:
        _TRAIN_STREAM = torch.cuda.Stream()
    return _TRAIN_STREAM


def _prep_train(case, seed):
    """A training run under way: moments of earlier steps, the step captured as a graph.  In
    the city each step takes other views of the pool, as a user samples them."""
    p, off, boxes, _ = _scene(case, seed)
    city = case["scene"] == "city"
    steps = [_cameras(case, seed, k) for k in range(2 if city else 1)]
    orders = [None if case["skip"] == "none" else orders_for_views(boxes, c) for c in steps]
    stream = _train_stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        cap = 16 * _pixels(case) if city else 0
        stp = BatchedStep(S.Context(), p, off, case["deg"], steps[0], None, S.opts(tile=case["tile"]),
                          pair_capacity=cap, stream=stream, order=orders[0], dssim=case["dssim"],
                          stale=case["skip"] == "stale")
        g = _gen(seed, 1)
        targets = [_uniform(g, stp.rgb.numel()) for _ in steps]
        scale = 1.0 / stp.rgb.numel()  # a loss gradient per colour value
        for k in GROUPS:
            stp.m[k].normal_(generator=g).mul_(0.1 * scale)
            stp.v[k].normal_(generator=g).exp_().mul_(scale * scale)
        stp.step_dev.fill_(1000)
        for cams, order, tgt in zip(steps[::-1], orders[::-1], targets[::-1]):
            if city:
                stp.set_views(cams, order)
            stp.set_targets(tgt)
            stp.run()
            code, _ = stp.status()
            if code != S.OK:
                raise RuntimeError(f"pair capacity: status {code}")
        stp.capture()
    stream.synchronize()
    return {"case": case, "stp": stp, "steps": list(zip(steps, orders, targets)) if city else None, "at": 0}


def _prep_render(case, seed):
    p, off, boxes, _ = _scene(case, seed)
    cams = _cameras(case, seed)
    b = S.Batch(S.Context(), _subsets(p, off, case["deg"]), cams, S.opts(tile=case["tile"]))
    if case["skip"] == "waves":
        b.set_order(orders_for_views(boxes, cams))
    return {"case": case, "keep": p, "b": b, "rgb": torch.empty(b.rgb_off[-1], device="cuda"),
            "T": torch.empty(b.total_pixels, device="cuda")}


def _prep_serve(case, seed):
    p, off, boxes, _ = _scene(case, seed)
    srv = S.Server(S.Context(), _subsets(p, off, case["deg"]), S.opts(tile=case["tile"]), 60 << 30,
                   slots=4, max_views=8)
    reqs = serve.poisson_requests(case["requests"], 200.0, seed, (0.0, 0.0, 0.0), 25.0)
    # the resolutions asked for go round, so that equal bursts ask for equal work
    cams = [I.pinhole(*RESOLUTIONS[i % 4], 60.0, r.cam.eye, (0.0, 0.0, 0.0)) for i, r in enumerate(reqs)]
    torch.cuda.synchronize()  # the server's own streams read the scene
    return {"case": case, "keep": p, "srv": srv, "boxes": boxes,
            "reqs": [serve.Request(r.arrival, c) for r, c in zip(reqs, cams)]}


def _prep_dssim(case, seed):
    g = _gen(seed)
    target = torch.nn.functional.interpolate(_uniform(g, 1, 3, max(2, case["h"] // 8), max(2, case["w"] // 8)),
                                             size=(case["h"], case["w"]), mode="bilinear")[0].contiguous()
    img = (target + 0.1 * _normal(g, 3, case["h"], case["w"])).clamp_(0.0, 1.0)
    return {"case": case, "ctx": S.Context(), "img": img, "target": target, "dL": torch.empty_like(img),
            "loss": torch.zeros(1, device="cuda")}


def _prep_adam(case, seed):
    n, deg, g = case["n"], case["deg"], _gen(seed)
    p = {"means": _uniform(g, n, 3, lo=-10.0, hi=10.0), **_attributes(g, n, deg, -3.0)}
    grad = {k: _normal(g, *v.shape) * 1e-6 for k, v in p.items()}
    m = {k: _normal(g, *v.shape) * 1e-7 for k, v in p.items()}
    v = {k: (_normal(g, *v.shape) * 1e-6).square_().add_(1e-14) for k, v in p.items()}
    return {"case": case, "ctx": S.Context(), "t": (p, grad, m, v), "hp": S.adam_hp(DEFAULT_LR),
            "structs": [S.params(*(d[k] for k in GROUPS), deg) for d in (p, grad, m, v)],
            "step": torch.full((1,), 1000, dtype=torch.int64, device="cuda")}


def _prep_composite(case, seed):
    """Partial images of K subsets, each covering a rectangle of the view."""
    g, rng, K, h, w = _gen(seed), np.random.default_rng(seed), case["K"], case["h"], case["w"]
    parts = []
    for _ in range(K):
        T = torch.ones(h, w, device="cuda")
        x0, y0 = int(rng.integers(0, w // 2 + 1)), int(rng.integers(0, h // 2 + 1))
        x1, y1 = int(rng.integers(x0, w)) + 1, int(rng.integers(y0, h)) + 1
        T[y0:y1, x0:x1] = _uniform(g, y1 - y0, x1 - x0, lo=1e-4, hi=1.0)
        parts.append({"rgb": _uniform(g, 3, h, w) * (1.0 - T), "T": T,
                      "depth": (1.0 - T) * _uniform(g, h, w, lo=2.0, hi=40.0),
                      "last": torch.zeros(h, w, dtype=torch.int32, device="cuda")})
    return {"case": case, "ctx": S.Context(), "parts": parts, "opts": S.opts(bg=(0.1, 0.2, 0.3)),
            "rgb": torch.empty(3, h, w, device="cuda"), "T": torch.empty(h, w, device="cuda")}


# ---------------------------------------------------------------- run
def run(state):
    return _RUN[state["case"]["kind"]](state)


def _run_partial(s):
    S.render_partial(s["ctx"], s["sub"], s["cam"], s["opts"], s["out"], keep_state=False)
    return s["out"]


def _run_noalloc(s):
    S.render_partial_noalloc(s["sub"], s["cam"], s["opts"], s["out"])
    return s["out"]


def _run_autograd(s):
    for v in s["p"].values():
        v.grad = None
    rgb, T = s["r"].render()
    loss = (rgb - s["target"]).abs().mean()
    loss.backward()
    return {"rgb": rgb, "T": T, "grads": {k: v.grad for k, v in s["p"].items()}}


def _run_view(s):
    c, ctx, o = s["case"], s["ctx"], s["opts"]
    for v in s["g"].values():
        v.zero_()
    states = [S.render_partial(ctx, sub, s["cam"], o, part) for sub, part in zip(s["subs"], s["parts"])]
    S.composite(ctx, s["parts"], c["w"], c["h"], o, s["img"])
    S.loss_l1(ctx, s["img"], s["target"], s["loss"], s["dL"])
    S.backward(ctx, s["subs"], s["cam"], s["parts"], states, s["dL"], None, o, s["grads"])
    for st in states:
        st.close()
    return {"img": s["img"], "loss": s["loss"], "grads": s["g"]}


def _run_train(s):
    stp = s["stp"]
    with torch.cuda.stream(stp.stream):
        if s["steps"]:
            cams, order, target = s["steps"][s["at"] % len(s["steps"])]
            s["at"] += 1
            stp.set_views(cams, order)
            stp.set_targets(target)
        stp.replay()
    return {"loss": stp.loss, "p": stp.p}


def _run_render(s):
    s["b"].forward(s["rgb"], s["T"])
    return {"rgb": s["rgb"], "T": s["T"]}


def _run_serve(s):
    boxes = s["boxes"]
    res = serve.run(s["srv"], s["reqs"], keep=set(range(len(s["reqs"]))), realtime=False,
                    order_fn=lambda c: front_to_back(boxes, c.eye))
    if res.failed:
        raise RuntimeError(f"{res.failed} requests failed")
    return [res.outputs[i] for i in range(res.n)]


def _run_dssim(s):
    S.loss_l1_dssim(s["ctx"], s["img"], s["target"], s["loss"], s["dL"], 0.2)
    return {"loss": s["loss"], "dL": s["dL"]}


def _run_adam(s):
    p, g, m, v = s["structs"]
    S.step_device(s["ctx"], p, g, m, v, s["hp"], s["step"])
    return {"p": s["t"][0], "m": s["t"][2], "v": s["t"][3]}


def _run_composite(s):
    c = s["case"]
    S.composite(s["ctx"], s["parts"], c["w"], c["h"], s["opts"], s["rgb"], s["T"])
    return {"rgb": s["rgb"], "T": s["T"]}


_PREPARE = {"partial": _prep_partial, "noalloc": _prep_partial, "autograd": _prep_autograd, "view": _prep_view,
            "train": _prep_train, "render": _prep_render, "serve": _prep_serve, "dssim": _prep_dssim,
            "adam": _prep_adam, "composite": _prep_composite}
_RUN = {"partial": _run_partial, "noalloc": _run_noalloc, "autograd": _run_autograd, "view": _run_view,
        "train": _run_train, "render": _run_render, "serve": _run_serve, "dssim": _run_dssim,
        "adam": _run_adam, "composite": _run_composite}


# ---------------------------------------------------------------- work
def work(case):
    """Bytes: parameters (and moments) read once, outputs written once.  Operations: a pixel
    blends some 100 Gaussians until it saturates (98 on the 10M-Gaussian views; fewer than
    the subsets' Gaussians can give), 18 operations each forward and 32 backward, plus about
    300 a Gaussian and view for the projection and as many for its adjoint."""
    kind = case["kind"]
    if kind == "dssim":  # two images in, one gradient out; two separable 11-tap windows
        px = 3 * case["w"] * case["h"]
        return {"bytes": 12 * px, "flops": px * (2 * 11 * 2 * 8 + 50)}
    if kind == "composite":
        px = case["w"] * case["h"]
        return {"bytes": px * (20 * case["K"] + 16), "flops": px * case["K"] * 10}
    per = 11 + 3 * I.n_sh_coeffs(case["deg"])
    if kind == "adam":  # p, g, m, v in; p, m, v out
        return {"bytes": 28 * per * case["n"], "flops": 14 * per * case["n"]}
    if kind == "serve":
        px = sum(RESOLUTIONS[i % 4][0] * RESOLUTIONS[i % 4][1] for i in range(case["requests"]))
        V = case["requests"]
    else:
        px, V = _pixels(case), case.get("views", 1)
    n = case["n"]
    blends = 100.0 * px
    fwd = blends * 18 + 300.0 * n * V
    bwd = blends * 32 + 300.0 * n * V
    if kind in ("partial", "noalloc"):
        return {"bytes": 4 * per * n + 24 * px, "flops": fwd}
    if kind in ("render", "serve"):
        return {"bytes": 4 * per * n + (16 if kind == "render" else 12) * px, "flops": fwd}
    if kind == "train":
        return {"bytes": 24 * per * n + 12 * px, "flops": fwd + bwd}
    return {"bytes": 8 * per * n + 28 * px, "flops": fwd + bwd}


# ---------------------------------------------------------------- 64 bits
def exact(case, seed):
    kind = case["kind"]
    if kind == "dssim":
        return _exact_dssim(case, seed)
    if kind == "adam":
        return _exact_adam(case, seed)
    if kind == "composite":
        s = _prep_composite(case, seed)
        C, T, D = (torch.stack([p[k] for p in s["parts"]]).double() for k in ("rgb", "T", "depth"))
        rgb, Tt = _composite64(C, T, D, torch.tensor([0.1, 0.2, 0.3], dtype=torch.float64, device="cuda"))
        return {"rgb": rgb, "T": Tt}
    if kind in ("partial", "noalloc") and case["n"] * case["w"] * case["h"] <= 2e10:
        p, _, _, _ = _scene(case, seed)
        with torch.no_grad():
            rgb, T, D = _partial64({k: v.double() for k, v in p.items()}, _cameras(case, seed)[0], case["deg"])
        return {"rgb": rgb, "T": T, "depth": D, "last": None}
    if kind == "autograd" and case["n"] * _pixels(case) <= 4e9:
        return _exact_autograd(case, seed)
    return None


def _exact_dssim(case, seed):
    s = _prep_dssim(case, seed)
    x, y = s["img"].double().requires_grad_(), s["target"].double()
    t = torch.arange(11, dtype=torch.float64, device="cuda") - 5
    w = torch.exp(-t * t / (2 * 1.5 * 1.5))
    w = w / w.sum()

    def blur(a):
        a = torch.nn.functional.pad(a[:, None], (5, 5, 5, 5))
        h = sum(w[k] * a[..., k:a.shape[-1] - 10 + k] for k in range(11))
        return sum(w[k] * h[..., k:h.shape[-2] - 10 + k, :] for k in range(11))[:, 0]
    mx, my = blur(x), blur(y)
    vx, vy, cov = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = ((2 * mx * my + c1) * (2 * cov + c2) / ((mx * mx + my * my + c1) * (vx + vy + c2))).mean()
    loss = 0.8 * (x - y).abs().mean() + 0.2 * (1 - ssim)
    loss.backward()
    return {"loss": loss.detach().reshape(1), "dL": x.grad}


def _exact_adam(case, seed):
    s = _prep_adam(case, seed)
    P, G, M, V = ({k: t.double() for k, t in d.items()} for d in s["t"])
    step, b1, b2, eps = 1001, 0.9, 0.999, 1e-15
    out = {"p": {}, "m": {}, "v": {}}
    for i, k in enumerate(GROUPS):
        lr = torch.full_like(P[k], DEFAULT_LR[i])
        if k == "sh":
            lr[:, 1:] = DEFAULT_LR[5]
        m = b1 * M[k] + (1 - b1) * G[k]
        v = b2 * V[k] + (1 - b2) * G[k] ** 2
        out["m"][k], out["v"][k] = m, v
        out["p"][k] = P[k] - lr * (m / (1 - b1 ** step)) / ((v / (1 - b2 ** step)).sqrt() + eps)
    return out


def _sh_basis(d, deg):
    x, y, z = d.unbind(-1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if deg >= 1:
        k = math.sqrt(3 / (4 * pi))
        Y += [-k * y, k * z, -k * x]
    if deg >= 2:
        k = math.sqrt(15 / (4 * pi))
        Y += [k * x * y, -k * y * z, math.sqrt(5 / (16 * pi)) * (3 * z * z - 1), -k * x * z,
              0.5 * k * (x * x - y * y)]
    if deg >= 3:
        k, q, r = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi)), math.sqrt(21 / (32 * pi))
        Y += [-k * y * (3 * x * x - y * y), q * x * y * z, -r * y * (5 * z * z - 1),
              math.sqrt(7 / (16 * pi)) * z * (5 * z * z - 3), -r * x * (5 * z * z - 1),
              0.5 * q * z * (x * x - y * y), -k * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


def _project64(p, cam, deg):
    """What one view keeps of a subset, front to back: 2-D mean, conic, pixel rectangle,
    opacity, depth, colour (EWA projection with 0.3 px^2 dilation)."""
    R = torch.from_numpy(np.asarray(cam.R, np.float64)).cuda()
    t = torch.from_numpy(np.asarray(cam.t, np.float64)).cuda()
    fx, fy, W, H = cam.fx, cam.fy, cam.width, cam.height
    cx, cy = cam.cx, cam.cy
    q = p["quats"] / p["quats"].norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    Rq = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                      2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                      2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).view(-1, 3, 3)
    V = R @ (Rq * p["log_scales"].exp()[:, None, :])
    c = p["means"] @ R.T + t
    tz = c[:, 2]
    lx, ly = 0.65 * W / fx, 0.65 * H / fy
    rx, ry = (c[:, 0] / tz).clamp(-lx, lx), (c[:, 1] / tz).clamp(-ly, ly)
    P0 = (fx / tz)[:, None] * V[:, 0] - (fx * rx / tz)[:, None] * V[:, 2]
    P1 = (fy / tz)[:, None] * V[:, 1] - (fy * ry / tz)[:, None] * V[:, 2]
    a, b, d = (P0 * P0).sum(1) + 0.3, (P0 * P1).sum(1), (P1 * P1).sum(1) + 0.3
    det = a * d - b * b
    mid = 0.5 * (a + d)
    rad = (3 * (mid + (mid * mid - det).clamp_min(0.1).sqrt()).sqrt()).ceil().detach()
    u, v = fx * c[:, 0] / tz + cx, fy * c[:, 1] / tz + cy
    eye = torch.from_numpy(cam.eye).cuda()
    dirs = p["means"] - eye
    Y = _sh_basis(dirs / dirs.norm(dim=1, keepdim=True), deg)
    col = ((Y[:, :, None] * p["sh"]).sum(1) + 0.5).clamp_min(0.0)
    keep = (tz > cam.near) & (det > 0) & (u + rad > 0) & (u - rad < W) & (v + rad > 0) & (v - rad < H)
    idx = torch.nonzero(keep).flatten()
    idx = idx[torch.argsort(tz[idx].detach(), stable=True)]
    o = torch.sigmoid(p["opacity_logits"])
    return [f[idx] for f in (u, v, d / det, -b / det, a / det, rad, o, tz)] + [col[idx]]


def _blend64(f, px, py, eps_T=1e-4):
    """Front-to-back blend of the projected Gaussians f at the pixels (px, py)."""
    u, v, A, B, C, rad, o, tz, col = f
    ud, vd = u.detach(), v.detach()
    dx, dy = px[:, None] + 0.5 - u, py[:, None] + 0.5 - v
    e = torch.exp(-0.5 * (A * dx * dx + 2 * B * dx * dy + C * dy * dy))
    al = (o * e).clamp_max(0.99)
    ins = ((px[:, None] + 0.5 >= ud - rad) & (px[:, None] + 0.5 <= ud + rad) &
           (py[:, None] + 0.5 >= vd - rad) & (py[:, None] + 0.5 <= vd + rad))
    al = torch.where(ins & (al >= 1.0 / 255.0), al, torch.zeros((), dtype=al.dtype, device=al.device))
    Ti = torch.cumprod(1 - al, dim=1)  # transmittance after each Gaussian
    al = torch.where(Ti.detach() >= eps_T, al, torch.zeros((), dtype=al.dtype, device=al.device))
    Ti = torch.cumprod(1 - al, dim=1)
    before = torch.cat([torch.ones_like(Ti[:, :1]), Ti[:, :-1]], 1)
    w = al * before
    T = Ti[:, -1] if Ti.shape[1] else torch.ones_like(px, dtype=torch.float64)
    return w @ col, T, w @ tz


def _partial64(p, cam, deg):
    f = _project64(p, cam, deg)
    H, W = cam.height, cam.width
    px = torch.arange(W, device="cuda", dtype=torch.float64).repeat(H)
    py = torch.arange(H, device="cuda", dtype=torch.float64).repeat_interleave(W)
    step = max(1, int(6e7) // max(1, f[0].numel()))
    got = [_blend64(f, px[i:i + step], py[i:i + step]) for i in range(0, px.numel(), step)]
    rgb, T, D = (torch.cat([g[k] for g in got]) for k in range(3))
    return rgb.T.reshape(3, H, W), T.view(H, W), D.view(H, W)


def _composite64(C, T, D, bg, eps=1e-4):
    """Eq. 5: C [K, 3, ...], T and D [K, ...]; subsets by D / (1 - T), empty ones last."""
    key = torch.where(T < 1, D / (1 - T).clamp_min(1e-300), torch.full_like(T, math.inf)).detach()
    order = torch.argsort(key, dim=0, stable=True)
    Ts = T.gather(0, order)
    Cs = C.gather(0, order[:, None].expand_as(C))
    P, rgb = torch.ones_like(T[0]), torch.zeros_like(C[0])
    for j in range(T.shape[0]):
        go = P.detach() >= eps
        rgb = rgb + torch.where(go, P, torch.zeros_like(P)) * Cs[j]
        P = torch.where(go, P * Ts[j], P)
    return rgb + bg.view(3, *([1] * (rgb.dim() - 1))) * P, P


def _exact_autograd(case, seed):
    p, off, _, _ = _scene(case, seed)
    p = {k: v.double().requires_grad_() for k, v in p.items()}
    cams, target = _cameras(case, seed), _uniform(_gen(seed, 1), 3 * _pixels(case)).double()
    bg = torch.zeros(3, dtype=torch.float64, device="cuda")
    total = float(target.numel())
    rgbs, Ts, at = [], [], 0
    for cam in cams:
        H, W = cam.height, cam.width
        fs = [_project64({k: v[int(off[i]):int(off[i + 1])] for k, v in p.items()}, cam, case["deg"])
              for i in range(len(off) - 1)]
        leaf = [[t.detach().requires_grad_() for t in f] for f in fs]
        tgt = target[at:at + 3 * H * W].view(3, H * W)
        at += 3 * H * W
        rgb, T = torch.empty(3, H * W, dtype=torch.float64, device="cuda"), torch.empty(H * W, dtype=torch.float64, device="cuda")
        step = max(1, int(1e7) // max(1, sum(f[0].numel() for f in fs)))
        for i in range(0, H * W, step):
            q = torch.arange(i, min(i + step, H * W), device="cuda")
            px, py = (q % W).double(), (q // W).double()
            parts = [_blend64(f, px, py) for f in leaf]
            C, Tk, D = torch.stack([a[0].T for a in parts]), torch.stack([a[1] for a in parts]), torch.stack([a[2] for a in parts])
            out, Tt = _composite64(C, Tk, D, bg)
            ((out - tgt[:, i:i + step]).abs().sum() / total).backward()
            rgb[:, i:i + step], T[i:i + step] = out.detach(), Tt.detach()
        back = [(t, l.grad) for f, lf in zip(fs, leaf) for t, l in zip(f, lf) if t.requires_grad and l.grad is not None]
        torch.autograd.backward([t for t, _ in back], [g for _, g in back])
        rgbs.append(rgb.reshape(-1))
        Ts.append(T)
    return {"rgb": torch.cat(rgbs), "T": torch.cat(Ts), "grads": {k: v.grad for k, v in p.items()}}
