"""Workloads by which the framework's speed is measured.

Each case is a plain dict; `prepare` makes what a user's program has in hand
before the call (a scene of surfels, a camera, targets, the buffers such a
program keeps), `run` is one pass through the public entry points and returns
all that the pass computes, `work` is the least a pass has to move and
compute, and `exact` is the same result in 64 bits, written from the
definitions in plain torch.
"""
import math
import random

import torch

from paper_2411_00771_gb300 import binding as B
from paper_2411_00771_gb300 import synthetic as syn
from paper_2411_00771_gb300 import training as T

DEV = "cuda"
PARAMS = ("mu", "quat", "scale", "opacity", "sh")
WEIGHTS = (0.8, 0.2, 0.5)  # L1, 1 - SSIM, inverse depth
# learning rates of a late training phase: repeated passes stay the same step
LATE_LR = dict(mu=1.6e-6, quat=1e-6, scale=1e-6, opacity=1e-6, sh=1e-6)
RESOLUTIONS = ((256, 256), (800, 600), (1600, 900), (1920, 1080), (3840, 2160))


def listed():
    return [
        # the small random scene: a quick check, a unit test, an interactive fit; launches and latency count
        dict(name="view_small", kind="view", scene="box", n=2000, width=128, height=128, sh=0, sets=1),
        # the headline step: one view of the aerial city block with loss, backward and Eq. 2 statistics
        dict(name="view_city_1m", kind="view", scene="city", n=1_000_000, width=1600, height=900, sh=3, sets=3),
        # one view of a lower-degree scene through torch.autograd, every loss term, an image of odd size
        dict(name="view_autograd_odd", kind="autograd", scene="city", n=600_000, width=1237, height=701, sh=2),
        # the training step of a large block: 4 views, every loss term, Adam
        dict(name="train_4m", kind="train", scene="city", n=4_000_000, width=1600, height=900, sh=3, views=4),
        # a thumbnail of a large scene: few tiles, long lists
        dict(name="render_256_4m", kind="render", scene="city", n=4_000_000, width=256, height=256, sh=3, half=False),
        # a full-HD frame of a fly-through
        dict(name="render_1080p_4m", kind="render", scene="city", n=4_000_000, width=1920, height=1080, sh=3,
             half=False),
        # a 4K frame of a compressed (vector-quantised, binary16) model
        dict(name="render_4k_8m_half", kind="render", scene="city", n=8_000_000, width=3840, height=2160, sh=3,
             half=True),
        # a burst of requests of all resolutions at the render server
        dict(name="serve_burst", kind="serve", scene="city", n=2_000_000, sh=3, requests=15),
        # the photometric and depth loss by itself
        dict(name="loss_900p", kind="loss", width=1600, height=900, depth=True, sets=3),
        # the trim contribution of one training view
        dict(name="contribution_1m", kind="contribution", scene="city", n=1_000_000, width=1600, height=900, sh=3,
             gamma=0.5),
        # the codebook of a compressed model
        dict(name="kmeans_2m", kind="kmeans", n=2_000_000, sh=3, K=8192, iters=10, keep=0.6),
        # visible frequency of the points of a block over its training views
        dict(name="visibility_8m", kind="visibility", n=8_000_000, width=1920, height=1080, views=300),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["view", "view", "autograd", "train", "render", "render", "serve", "loss", "contribution",
                       "kmeans", "visibility"])
    sh = rng.choice([0, 1, 2, 3, 3, 3])
    if kind == "loss":
        return dict(kind=kind, width=_log(rng, 64, 3840), height=_log(rng, 48, 2160), depth=rng.random() < 0.7,
                    sets=rng.choice([1, 3]))
    if kind == "kmeans":
        return dict(kind=kind, n=_log(rng, 20_000, 2_000_000), sh=sh, K=rng.choice([512, 1000, 2048, 4096, 8192]),
                    iters=rng.randint(1, 10), keep=round(rng.uniform(0.5, 0.8), 3))
    if kind == "visibility":
        return dict(kind=kind, n=_log(rng, 50_000, 8_000_000), width=_log(rng, 640, 3840), height=_log(rng, 480, 2160),
                    views=rng.randint(20, 300))
    if kind == "serve":
        return dict(kind=kind, scene="city", n=_log(rng, 100_000, 2_000_000), sh=sh, requests=rng.randint(4, 15))
    if kind == "view" and rng.random() < 0.3:
        return dict(kind=kind, scene="box", n=_log(rng, 300, 20_000), width=_log(rng, 33, 400),
                    height=_log(rng, 33, 300), sh=sh, sets=rng.choice([1, 3]))
    c = dict(kind=kind, scene="city", n=_log(rng, 50_000, 4_000_000), width=_log(rng, 200, 1920),
             height=_log(rng, 150, 1080), sh=sh)
    if kind == "view":
        c.update(n=min(c["n"], 2_000_000), sets=rng.choice([1, 3, 3]))
    elif kind == "train":
        c.update(views=rng.randint(1, 4))
    elif kind == "render":
        c.update(half=rng.random() < 0.3)
    elif kind == "contribution":
        c.update(gamma=rng.choice([0.0, 0.5, 0.5, 1.0]))
    return c


# ---------------------------------------------------------------------------
# Inputs, drawn on the GPU.

def _rand(g, *shape):
    return torch.rand(shape, device=DEV, generator=g)


def _randn(g, *shape):
    return torch.randn(shape, device=DEV, generator=g)


def _uniform(g, a, b, *shape):
    return a + (b - a) * _rand(g, *shape)


def _box_scene(g, n, deg):
    """Surfels scattered in front of a pinhole camera, sizes over two octaves, any orientation."""
    mu = torch.stack([_uniform(g, -1, 1, n), _uniform(g, -1, 1, n), _uniform(g, 2, 4, n)], 1)
    q = _randn(g, n, 4)
    P = dict(mu=mu, quat=q / q.norm(dim=1, keepdim=True), scale=torch.exp(_uniform(g, -4, -2, n, 2)),
             opacity=torch.sigmoid(_randn(g, n)), sh=0.05 * _randn(g, n, (deg + 1) ** 2, 3))
    P["sh"][:, 0] = _uniform(g, -math.sqrt(math.pi), math.sqrt(math.pi), n, 3)
    return P


def _city_points(g, n, side=14, extent=500.0):
    """Points by area on the ground, roofs and walls of a block of side x side box buildings:
    (points, index of the face's normal, colour)."""
    cell = extent / side
    nb = side * side
    half = _uniform(g, 5.0, 0.4 * cell, nb, 2)
    mid = (torch.stack(torch.meshgrid(torch.arange(side, device=DEV), torch.arange(side, device=DEV), indexing="ij"),
                       -1).reshape(nb, 2) + 0.5) * cell - extent / 2
    h = _uniform(g, 10.0, 60.0, nb)
    albedo = _uniform(g, 0.2, 0.85, nb, 3)
    walls = torch.stack([half[:, 1] * h, half[:, 1] * h, half[:, 0] * h, half[:, 0] * h]) * 2  # [4, nb]
    area = extent * extent + float(walls.sum())
    on_wall = _rand(g, n) < float(walls.sum()) / area
    # ground and roofs: a point over a footprint lies on the roof
    xy = (_rand(g, n, 2) - 0.5) * extent
    ij = ((xy + extent / 2) / cell).long().clamp_(0, side - 1)
    b = ij[:, 0] * side + ij[:, 1]
    roof = ((xy - mid[b]).abs() < half[b]).all(1)
    mu = torch.cat([xy, torch.where(roof, h[b], torch.zeros_like(h[b]))[:, None]], 1)
    face = torch.zeros(n, dtype=torch.long, device=DEV)
    col = torch.where(roof[:, None], 0.8 * albedo[b], torch.tensor([0.45, 0.47, 0.42], device=DEV))
    # walls
    cum = torch.cumsum(walls.reshape(-1).double(), 0)
    wall = torch.searchsorted(cum, _rand(g, n).double() * cum[-1]).clamp_(max=4 * nb - 1)
    wf, wb = wall // nb, wall % nb
    sign = torch.where(wf % 2 == 0, 1.0, -1.0)
    along = _uniform(g, -1, 1, n)
    u = torch.where(wf < 2, sign, along) * half[wb, 0] + mid[wb, 0]
    v = torch.where(wf < 2, along, sign) * half[wb, 1] + mid[wb, 1]
    wmu = torch.stack([u, v, _rand(g, n) * h[wb]], 1)
    w = on_wall[:, None]
    return torch.where(w, wmu, mu), torch.where(on_wall, wf + 1, face), torch.where(w, albedo[wb], col), area


def _city_scene(g, n, deg):
    """Surfels on the surfaces of a 500 m city block: local z the surface normal, sizes about half the
    spacing, one in twenty elongated."""
    mu, face, col, area = _city_points(g, n)
    # quaternions that take z to +z, +x, -x, +y, -y, after a spin about z
    r = math.sqrt(0.5)
    base = torch.tensor([[1, 0, 0, 0], [r, 0, r, 0], [r, 0, -r, 0], [r, -r, 0, 0], [r, r, 0, 0]], device=DEV)[face]
    a = _uniform(g, 0, math.pi, n)
    c, s = torch.cos(a), torch.sin(a)
    w, x, y, z = base.unbind(1)
    quat = torch.stack([w * c - z * s, x * c + y * s, y * c - x * s, z * c + w * s], 1)
    spacing = math.sqrt(area / n)
    log_s = math.log(0.5 * spacing) + 0.4 * _randn(g, n, 2)
    long = (_rand(g, n) < 0.05)[:, None] & (torch.arange(2, device=DEV)[None] == (_rand(g, n) < 0.5).long()[:, None])
    log_s = log_s + torch.where(long, _uniform(g, math.log(10), math.log(50), n, 2), torch.zeros_like(log_s))
    sh = 0.05 * _randn(g, n, (deg + 1) ** 2, 3)
    sh[:, 0] = ((col + 0.05 * _randn(g, n, 3)).clamp(0, 1) - 0.5) * 2 * math.sqrt(math.pi)
    return dict(mu=mu.contiguous(), quat=quat.contiguous(), scale=torch.exp(log_s), sh=sh.contiguous(),
                opacity=torch.sigmoid(1 + 1.5 * _randn(g, n)))


def _make(case, g):
    return (_box_scene if case["scene"] == "box" else _city_scene)(g, case["n"], case["sh"])


def _camera(case, rng):
    if case.get("scene") == "box":
        return syn.identity_camera(case["width"], case["height"], 128.0)
    return _orbit(rng, case["width"], case["height"])


def _orbit(rng, W, H):
    az, r = rng.uniform(0, 2 * math.pi), rng.uniform(150.0, 250.0)
    tgt = (rng.uniform(-60, 60), rng.uniform(-60, 60), 0.0)
    pos = (tgt[0] + r * math.cos(az), tgt[1] + r * math.sin(az), rng.uniform(140.0, 200.0))
    return syn.look_at(pos, tgt, W, H, 0.5 * W / math.tan(math.radians(30.0)))


def _targets(g, P, deg, cam):
    """Colour and inverse depth of the view that training is to reach: a render of the scene with its
    colours, opacities and places a little off, and the noise of a photograph."""
    Q = {k: v.clone() for k, v in P.items()}
    Q["sh"][:, 0] += 0.3 * _randn(g, *Q["sh"][:, 0].shape)
    Q["mu"] += 0.2 * Q["scale"].mean(1, keepdim=True) * _randn(g, *Q["mu"].shape)
    Q["opacity"] = torch.sigmoid(torch.logit(Q["opacity"].clamp(1e-4, 1 - 1e-4)) + 0.3 * _randn(g, len(Q["opacity"])))
    sc = B.Scene(*[Q[k] for k in PARAMS], deg)
    out, _ = sc.render(cam, save=False)
    torch.cuda.synchronize()
    sc.close()
    tgt = (out[:3] + 0.02 * _randn(g, 3, cam["height"], cam["width"])).clamp_(0, 1)
    return tgt.contiguous(), (out[5] / out[3].clamp_min(1e-3)).contiguous()


def prepare(case, seed):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    rng = random.Random(int(seed))
    kind, s = case["kind"], dict(case=case)
    if kind == "loss":
        H, W = case["height"], case["width"]
        # a smooth image and its noisy target
        low = torch.nn.functional.interpolate(_rand(g, 1, 3, H // 16 + 2, W // 16 + 2), size=(H, W), mode="bilinear")[0]
        out = torch.zeros((12, H, W), device=DEV)
        out[:3] = low + 0.03 * _randn(g, 3, H, W)
        out[5] = _uniform(g, 0.003, 0.007, H, W)
        s.update(out=out, target=(low + 0.05 * _randn(g, 3, H, W)).clamp_(0, 1),
                 tinv=_uniform(g, 0.003, 0.007, H, W) if case["depth"] else None,
                 adj=[torch.zeros((11, H, W), device=DEV) for _ in range(case["sets"])],
                 losses=torch.empty(4, device=DEV))
        return s
    if kind == "kmeans":
        # trained SH: a base colour of its surface, noise, small higher orders
        n, K = case["n"], (case["sh"] + 1) ** 2
        base = (_uniform(g, 0.2, 0.85, 200, 3) - 0.5) * 2 * math.sqrt(math.pi)
        sh = 0.05 * _randn(g, n, K, 3)
        sh[:, 0] = base[torch.randint(0, 200, (n,), device=DEV, generator=g)] + 0.17 * _randn(g, n, 3)
        s.update(sh=sh, keep=(_rand(g, n) < case["keep"]).to(torch.uint8), u=_rand(g, case["K"]))
        return s
    if kind == "visibility":
        s.update(points=(_city_points(g, case["n"])[0]
                         + 0.25 * (_rand(g, case["n"], 3) - 0.5)).contiguous(),
                 cams=[_orbit(rng, case["width"], case["height"]) for _ in range(case["views"])])
        return s
    P = _make(case, g)
    n, deg = case["n"], case["sh"]
    s["P"] = P
    if kind == "serve":
        s["scene"] = B.Scene(*[P[k] for k in PARAMS], deg)
        s["server"] = B.Server(24 << 30)
        s["id"] = s["server"].add_scene(s["scene"])
        s["cams"] = [_orbit(rng, *RESOLUTIONS[i % len(RESOLUTIONS)]) for i in range(case["requests"])]
        s["outs"] = [torch.empty((12, c["height"], c["width"]), device=DEV) for c in s["cams"]]
        torch.cuda.synchronize()  # the server's streams do not wait for this one
        return s
    if kind == "train":
        s["views"] = []
        for _ in range(case["views"]):
            cam = _camera(case, rng)
            s["views"].append((cam, *_targets(g, P, deg, cam)))
        s["trainer"] = T.Trainer(P["mu"], P["quat"], torch.log(P["scale"]),
                                 torch.logit(P["opacity"].clamp(1e-6, 1 - 1e-6)), P["sh"], deg, lr=LATE_LR,
                                 w_dist=0.01)
        return s
    cam = s["cam"] = _camera(case, rng)
    H, W = cam["height"], cam["width"]
    if kind == "render" and case["half"]:
        # the codebook's quality does not matter to the render: two steps of K-means
        contrib = _rand(g, n)
        comp, _ = B.compress(tuple(P[k] for k in PARAMS), deg, contrib, 0.4, 2048, 2, _rand(g, 2048))
        s["scene"] = B.CompressedScene(comp)
        del s["P"]
        return s
    s["scene"] = B.Scene(*[P[k] for k in PARAMS], deg)
    if kind == "contribution":
        s["contrib"], s["sum"] = torch.zeros(n, device=DEV), torch.zeros(n, device=DEV)
        s["count"] = torch.zeros(n, dtype=torch.int32, device=DEV)
    if kind in ("view", "autograd"):
        s["target"], s["tinv"] = _targets(g, P, deg, cam)
    if kind == "autograd":
        for v in P.values():
            v.requires_grad_(True)
    if kind == "view":
        s["out"] = torch.empty((12, H, W), device=DEV)
        s["adj"] = [torch.zeros((11, H, W), device=DEV) for _ in range(case["sets"])]
        s["grads"] = {k: torch.zeros_like(v) for k, v in P.items()}
        s["losses"] = torch.empty(4, device=DEV)
        if case["sets"] == 3:
            s["screen"] = torch.zeros((3, n, 2), device=DEV)
            s["stats"] = torch.zeros((n, 4), device=DEV)
    return s


# ---------------------------------------------------------------------------
# One pass.

def run(s):
    case = s["case"]
    return globals()["_run_" + case["kind"]](s, case)


def _run_view(s, case):
    sc, adj = s["scene"], s["adj"]
    three = case["sets"] == 3
    out, frame = sc.render(s["cam"], out=s["out"])
    B.loss(out, s["target"], s["tinv"], WEIGHTS, adj_total=adj[0], adj_ssim=adj[1] if three else None,
           adj_l1=adj[2] if three else None, losses=s["losses"])
    for v in s["grads"].values():
        v.zero_()
    masks = [0x7 | (1 << 5), 0x7, 0x7][:len(adj)]
    if not three:
        sc.backward(frame, adj, masks, s["grads"])
        frame.release()
        return {"out": out, "losses": s["losses"], "grads": s["grads"]}
    s["screen"].zero_()
    sc.backward(frame, adj, masks, s["grads"], s["screen"])
    sc.densify_accumulate(frame, s["screen"], s["stats"])
    # the mask is grad >= threshold, which rounding decides: grad and k are what is compared
    _, grad, k = B.densify_select(s["stats"], s["P"]["scale"])
    keep = B.elongation_filter(s["P"]["scale"])
    frame.release()
    return {"out": out, "losses": s["losses"], "grads": s["grads"], "screen": s["screen"], "stats": s["stats"],
            "grad": grad, "k": k, "keep": keep}


def _run_autograd(s, case):
    P = s["P"]
    for v in P.values():
        v.grad = None
    out = T.render(s["scene"], s["cam"], T.MASK_TRAIN, params=[P[k] for k in PARAMS])
    total, parts = T.loss(out, s["target"], s["tinv"], s["cam"], WEIGHTS, w_dist=0.01)
    total.backward()
    return {"out": out.detach(), "parts": parts, "grads": {k: v.grad for k, v in P.items()}}


def _run_train(s, case):
    tr = s["trainer"]
    losses = tr.step(s["views"])
    return {"losses": losses, "raw": tr.raw, "grads": tr.grads, "stats": tr.stats}


def _run_render(s, case):
    return s["scene"].render(s["cam"], save=False)[0]


def _run_serve(s, case):
    srv = s["server"]
    tickets = [srv.submit(s["id"], c, o) for c, o in zip(s["cams"], s["outs"])]
    for t in tickets:
        srv.wait(t)
    return s["outs"]


def _run_loss(s, case):
    adj = s["adj"] + [None, None]
    B.loss(s["out"], s["target"], s["tinv"], WEIGHTS if case["depth"] else (0.8, 0.2, 0.0), adj_total=adj[0],
           adj_ssim=adj[1], adj_l1=adj[2], losses=s["losses"])
    return {"adj": s["adj"], "losses": s["losses"]}


def _run_contribution(s, case):
    s["contrib"].zero_()
    s["scene"].contribution(s["cam"], gamma=case["gamma"], contrib=s["contrib"], view_sum=s["sum"],
                            view_count=s["count"])
    return {"contrib": s["contrib"], "sum": s["sum"], "count": s["count"]}


def _run_kmeans(s, case):
    cb, assign, obj, m = B.vq_kmeans(s["sh"], case["sh"], s["keep"], case["K"], case["iters"], s["u"])
    return {"codebook": cb, "assign": assign, "objective": obj, "m": m}


def _run_visibility(s, case):
    counts = B.visibility_count(s["points"], 0.1, s["cams"])
    keep, z = B.visibility_bounds(s["points"], counts, 3)
    return {"counts": counts, "keep": keep, "z": z}


# ---------------------------------------------------------------------------
# What a pass cannot do without.  Which surfels a view holds and how many of them a pixel blends
# depends on the scene; a quarter of a city block lies in a view, and a pixel blends about LAYERS.

LAYERS = 30
IN_VIEW = 0.25


def _view_work(n, pixels, deg, train):
    """Each surfel's place, turn and size is read (36 bytes), the rest of those in view (4 + 12 per SH
    coefficient), 12 planes written.  Backward: the planes' adjoints read, every gradient written once.
    Per pixel and blended surfel about 50 operations forward, 165 backward."""
    rest = 4 + 12 * (deg + 1) ** 2
    by = 36 * n + IN_VIEW * n * rest + 48 * pixels
    fl = 50 * LAYERS * pixels
    if train:
        by += IN_VIEW * n * (36 + rest) + n * (36 + rest) + 3 * 12 * pixels + 16 * pixels
        fl += 165 * LAYERS * pixels
    return by, fl


def work(case):
    kind = case["kind"]
    if kind == "kmeans":
        C = 3 * (case["sh"] + 1) ** 2
        m = (1 - case["keep"]) * case["n"]
        return {"bytes": case["n"] * 5 + m * 4 * C + 2 * case["K"] * C,
                "flops": 2.0 * m * case["K"] * C * (case["iters"] + 1)}
    if kind == "visibility":
        return {"bytes": case["n"] * 17, "flops": 35.0 * case["n"] * case["views"]}
    if kind == "serve":
        px = [RESOLUTIONS[i % len(RESOLUTIONS)] for i in range(case["requests"])]
        parts = [_view_work(case["n"], w * h, case["sh"], False) for w, h in px]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    px = case["width"] * case["height"]
    if kind == "loss":
        # five windowed moments forward, three backward, 2 x 11 taps each, for three channels
        return {"bytes": px * (24 + 12 * case["sets"] + (12 if case["depth"] else 0)),
                "flops": 3.0 * px * (8 * 44 + 60)}
    by, fl = _view_work(case["n"], px, case["sh"], kind in ("view", "autograd", "train"))
    if kind == "train":
        values = case["n"] * (10 + 3 * (case["sh"] + 1) ** 2)
        by, fl = case["views"] * by + 28 * values, case["views"] * fl + 12 * values
    if kind == "render" and case["half"]:
        by -= case["n"] * (12 + IN_VIEW * (2 + 6 * (case["sh"] + 1) ** 2))
    if kind == "contribution":
        by += 12 * case["n"] - 48 * px
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# The same in 64 bits, from the definitions: every surfel against every pixel.

def exact(case, seed):
    kind = case["kind"]
    if kind == "loss":
        s = prepare(case, seed)
        out = s["out"].double().requires_grad_(True)
        tinv = None if s["tinv"] is None else s["tinv"].double()
        w = WEIGHTS if case["depth"] else (0.8, 0.2, 0.0)
        parts = _loss64(out, s["target"].double(), tinv, w)
        tot, ssim, l1 = [torch.autograd.grad(x, out, retain_graph=True)[0][:11] for x in
                         (parts[3], w[1] * (1 - parts[1]), w[0] * parts[0])]
        return {"adj": [tot, ssim, l1][:case["sets"]], "losses": torch.stack(parts).detach()}
    if kind == "view" and case["scene"] == "box" and case["sets"] == 1:
        if case["n"] * case["width"] * case["height"] > 50_000_000:
            return None
        s = prepare(case, seed)
        leaf = {k: v.double().requires_grad_(True) for k, v in s["P"].items()}
        out = _render64(leaf, s["cam"], case["sh"])
        parts = _loss64(out, s["target"].double(), s["tinv"].double(), WEIGHTS)
        grads = torch.autograd.grad(parts[3], [leaf[k] for k in PARAMS], allow_unused=True)
        return {"out": out.detach(), "losses": torch.stack(parts).detach(),
                "grads": {k: torch.zeros_like(leaf[k]) if v is None else v for k, v in zip(PARAMS, grads)}}
    return None


def _blur64(x):
    k = torch.exp(-(torch.arange(11, device=x.device).double() - 5) ** 2 / (2 * 1.5 ** 2))
    k = k / k.sum()
    x = torch.nn.functional.pad(x, (5, 5, 5, 5))
    H, W = x.shape[-2] - 10, x.shape[-1] - 10
    x = sum(k[i] * x[..., i:i + W] for i in range(11))
    return sum(k[i] * x[..., i:i + H, :] for i in range(11))


def _loss64(out, tgt, tinv, w):
    x = out[:3]
    l1 = (x - tgt).abs().mean()
    mx, my = _blur64(x), _blur64(tgt)
    vx, vy, vxy = _blur64(x * x) - mx * mx, _blur64(tgt * tgt) - my * my, _blur64(x * tgt) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = ((2 * mx * my + c1) * (2 * vxy + c2) / ((mx * mx + my * my + c1) * (vx + vy + c2))).mean()
    depth = (out[5] - tinv).abs().mean() if tinv is not None else x.sum() * 0
    return [l1, ssim, depth, w[0] * l1 + w[1] * (1 - ssim) + w[2] * depth]


def _sh64(d, deg):
    """Real spherical harmonics with the Condon-Shortley phase, in the order of (l, m)."""
    x, y, z = d.unbind(1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if deg > 0:
        c = math.sqrt(3 / (4 * pi))
        Y += [-c * y, c * z, -c * x]
    if deg > 1:
        a, b, c = math.sqrt(15 / pi) / 2, math.sqrt(5 / pi) / 4, math.sqrt(15 / pi) / 4
        Y += [a * x * y, -a * y * z, b * (2 * z * z - x * x - y * y), -a * x * z, c * (x * x - y * y)]
    if deg > 2:
        a, b = math.sqrt(35 / (2 * pi)) / 4, math.sqrt(105 / pi) / 2
        c, e, f = math.sqrt(21 / (2 * pi)) / 4, math.sqrt(7 / pi) / 4, math.sqrt(105 / pi) / 4
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (4 * z * z - x * x - y * y),
              e * z * (2 * z * z - 3 * x * x - 3 * y * y), -c * x * (4 * z * z - x * x - y * y),
              f * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _render64(P, cam, deg):
    R = torch.as_tensor(cam["R"], dtype=torch.float64, device=DEV)
    t = torch.as_tensor(cam["t"], dtype=torch.float64, device=DEV)
    H, W, fx, fy = cam["height"], cam["width"], cam["fx"], cam["fy"]
    q = P["quat"] / P["quat"].norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    r1 = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + w * z), 2 * (x * z - w * y)], 1)
    r2 = torch.stack([2 * (x * y - w * z), 1 - 2 * (x * x + z * z), 2 * (y * z + w * x)], 1)
    r3 = torch.stack([2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y)], 1)
    p = P["mu"] @ R.T + t
    a, b = (r1 @ R.T) * P["scale"][:, :1], (r2 @ R.T) * P["scale"][:, 1:]
    nrm = r3 @ R.T
    nrm = nrm * torch.where((nrm * p).sum(1, keepdim=True) > 0, -1.0, 1.0)
    vis = (p[:, 2] - 3 * torch.sqrt(a[:, 2] ** 2 + b[:, 2] ** 2) > 0.2).nonzero()[:, 0]
    # front to back by the centre's depth as a 32-bit number, ties by index
    vis = vis[torch.sort(p[vis, 2].detach().float(), stable=True)[1]]
    p, a, b, nrm, opac, sh, mu = p[vis], a[vis], b[vis], nrm[vis], P["opacity"][vis], P["sh"][vis], P["mu"][vis]
    pz = p[:, 2]
    xi, yi = p[:, 0] / pz, p[:, 1] / pz
    cx, cy = fx * xi + cam["cx"], fy * yi + cam["cy"]
    J11, J12 = fx * (a[:, 0] - a[:, 2] * xi) / pz, fx * (b[:, 0] - b[:, 2] * xi) / pz
    J21, J22 = fy * (a[:, 1] - a[:, 2] * yi) / pz, fy * (b[:, 1] - b[:, 2] * yi) / pz
    det = J11 * J22 - J12 * J21
    i11, i12, i21, i22 = J22 / det, -J12 / det, -J21 / det, J11 / det
    w1, w2 = a[:, 2] / pz, b[:, 2] / pz
    e1, e2 = -(i11 * w1 + i21 * w2), -(i12 * w1 + i22 * w2)
    d = mu - (-R.T @ t)
    rgb = ((_sh64(d / d.norm(dim=1, keepdim=True), deg)[:, :, None] * sh).sum(1) + 0.5).clamp_min(0)
    jj, ii = torch.meshgrid(torch.arange(H, device=DEV).double() + 0.5, torch.arange(W, device=DEV).double() + 0.5,
                            indexing="ij")
    dx, dy = ii.reshape(-1, 1) - cx, jj.reshape(-1, 1) - cy  # [pixels, surfels]
    den = 1 + e1 * dx + e2 * dy
    u, v = (i11 * dx + i12 * dy) / den, (i21 * dx + i22 * dy) / den
    obj = u * u + v * v
    scr = 2 * (dx * dx + dy * dy)
    use = (den > 0) & (obj <= scr)
    rho = torch.where(use, obj, scr)
    alpha = (opac * torch.exp(-rho / 2)).clamp_max(0.99)
    alpha = torch.where((rho <= 9) & (alpha >= 1 / 255), alpha, torch.zeros_like(alpha))
    after = torch.cumprod(1 - alpha, 1)
    on = (alpha > 0) & (after.detach() >= 1e-4)
    alpha = torch.where(on, alpha, torch.zeros_like(alpha))
    after = torch.cumprod(1 - alpha, 1)
    front = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
    wt = alpha * front
    zz = torch.where(use, pz / den, pz.expand_as(den))
    zz = torch.where(on, zz, torch.ones_like(zz))
    A, Z = torch.cumsum(wt, 1), torch.cumsum(wt * zz, 1)
    dist = (2 * wt * (zz * (A - wt) - (Z - wt * zz))).sum(1)
    order = torch.where(on & (front > 0.5), torch.arange(1, len(vis) + 1, device=DEV), 0).max(1)[0]
    med = torch.where(order > 0, zz.gather(1, (order - 1).clamp_min(0)[:, None])[:, 0], torch.zeros_like(dist))
    planes = [wt @ rgb, A[:, -1:], Z[:, -1:], (wt / zz).sum(1, keepdim=True), med[:, None], wt @ nrm, dist[:, None],
              after[:, -1:]]
    return torch.cat(planes, 1).T.reshape(12, H, W)
