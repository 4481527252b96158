"""Edges of the blends: images that end inside a 4x4 block, a tile row or a
tile; lists that end on and beside the sizes in which they are staged; the
backward in several passes when memory is short; infinities and NaN in an
adjoint.  Against the FP64 oracle at the tolerances of the parity tests (2e-5
per channel, 1e-3 relative per gradient)."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2411_00771_gb300 import synthetic as syn
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

FLAG_ANY = oracle.FLAG_ALPHA | oracle.FLAG_RHO | oracle.FLAG_TSTOP | oracle.FLAG_MEDIAN


def _check(scene, cam, masks, seed, settings=None):
    sc, d, out, cnt, frame = gu.gpu_render(scene, cam, settings)
    ref = oracle.render(scene, cam, settings=settings)
    ok = (ref["flags"] & FLAG_ANY) == 0
    nb = ok & ((ref["flags"] & oracle.FLAG_BRANCH) == 0)
    v, vb = (gu.plane_violations(out.cpu().numpy(), ref["out"], m) for m in (ok, nb))
    for p, name in enumerate(gu.PLANES):
        assert (vb if p in gu.DEPTH_PLANES else v)[p] <= 1.0, name
    assert np.array_equal(cnt.cpu().numpy()[ok], ref["count"][ok])
    # a render that keeps no frame gives the same planes
    again, _ = sc.render(cam, save=False)
    assert torch.equal(again, out)
    H, W = cam["height"], cam["width"]
    rng = np.random.default_rng(seed)
    # adjoints only where the oracle saw no decision within a hair of its threshold
    adj = rng.normal(size=(len(masks), 11, H, W)) * nb
    for s, m in enumerate(masks):
        for p in range(11):
            if not (m >> p) & 1:
                adj[s, p] = 0.0
    n = scene["mu"].shape[0]
    grads = {k: torch.zeros_like(x) for k, x in d.items()}
    screen = torch.zeros((len(masks), n, 2), device="cuda")
    sc.backward(frame, [torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda() for a in adj], masks, grads,
                screen)
    torch.cuda.synchronize()
    r = oracle.backward(scene, cam, np.float32(adj).astype(np.float64), settings=settings)
    for k in grads:
        assert gu.rel_err(grads[k].cpu().numpy(), r[k].reshape(grads[k].shape)) <= 1e-3, k
    for s in range(len(masks)):
        assert gu.rel_err(screen[s].cpu().numpy(), r["screen"][s]) <= 1e-3, ("screen", s)


LOSS = [0x7 | (1 << 5), 0x7, 0x7]


@pytest.mark.parametrize("masks", [LOSS, [0x7FF], [0x7FF, 0x7, 0x7]], ids=["loss", "all", "all3"])
@pytest.mark.parametrize("W,H", [(1, 1), (3, 5), (16, 16), (17, 4), (21, 33), (34, 15)])
def test_image_ends_inside_a_block(W, H, masks):
    scene, cam, _, _ = syn.tiny_scene(seed=900 + W, n=400, width=W, height=H, fx=1.2 * max(W, H), sh_degree=1,
                                      log_scale_range=(-3.5, -1.5))
    _check(scene, cam, masks, seed=W * 100 + H, settings=dict(bg=(0.3, 0.6, 0.1)))


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 96, 128, 256, 257])
def test_list_lengths_around_the_staging_sizes(n):
    """n wide faint disks over one 16 x 16 tile: every 4 x 4 block's list has
    all n entries and no pixel stops."""
    rng = np.random.default_rng(n)
    q = rng.normal(0.0, 0.05, (n, 4))
    q[:, 0] = 1.0
    scene = dict(mu=np.column_stack([rng.uniform(-0.05, 0.05, (n, 2)), rng.uniform(2, 4, n)]).astype(np.float32),
                 quat=q.astype(np.float32), scale=rng.uniform(1.0, 1.5, (n, 2)).astype(np.float32),
                 opacity=rng.uniform(0.006, 0.02, n).astype(np.float32),
                 sh=rng.normal(0, 0.5, (n, 1, 3)).astype(np.float32), sh_degree=0)
    _check(scene, syn.identity_camera(16, 16, 16.0), LOSS, seed=n)
    _check(scene, syn.identity_camera(16, 16, 16.0), [0x7FF], seed=n + 1)


def _limited_scene(d, deg, limit):
    """A scene whose allocator refuses requests above limit[0] bytes."""
    from paper_2411_00771_gb300 import binding as B
    live, sizes = {}, []

    def alloc(size, ctx, stream):
        if size > limit[0]:
            return None
        t = torch.empty(size, dtype=torch.uint8, device="cuda")
        live[t.data_ptr()] = t
        sizes.append(size)
        return t.data_ptr()

    def free(ptr, size, ctx, stream):
        torch.cuda.synchronize()
        live.pop(ptr, None)

    desc = B.gs_scene_desc()
    desc.settings, desc.sh_degree = B.default_settings(), deg
    desc.allocator = B.gs_allocator(B.ALLOC_FN(alloc), B.FREE_FN(free), None)
    sc = B.Scene(*[d[k] for k in ("mu", "quat", "scale", "opacity", "sh")], deg)
    B._check(B.lib().gs_destroy_scene(sc._handle))
    sc._handle = ctypes.c_void_p()
    sc._fill(desc, *[d[k] for k in ("mu", "quat", "scale", "opacity", "sh")])
    B._check(B.lib().gs_create_scene(ctypes.byref(sc._handle), ctypes.byref(desc)))
    sc._keep = desc
    return sc, sizes


@pytest.mark.parametrize("masks", [LOSS, [0x7FF]], ids=["loss", "all"])
def test_backward_in_passes_when_memory_is_short(masks):
    """Rows for a part of the surfels at a time give the same gradients: each
    row's sum differs only in the order of additions in double, so 1e-6
    relative (a few roundings to float) bounds the difference."""
    scene, cam, _, _ = syn.tiny_scene(seed=55, n=3000, width=96, height=80, fx=90.0, sh_degree=2)
    d = gu.to_dev(scene)
    limit = [1 << 40]
    sc, sizes = _limited_scene(d, 2, limit)
    out, frame = sc.render(cam)
    rng = np.random.default_rng(3)
    adj = [torch.from_numpy(rng.normal(size=(11, 80, 96)).astype(np.float32)).cuda() for _ in masks]
    res = []
    for cap in (1 << 40, 64 * 3000, 20_000):
        limit[0] = cap
        g = {k: torch.zeros_like(v) for k, v in d.items()}
        screen = torch.zeros((len(masks), 3000, 2), device="cuda")
        sc.backward(frame, adj, masks, g, screen)
        torch.cuda.synchronize()
        assert sizes[-1] <= cap
        res.append({**g, "screen": screen})
    limit[0] = 1 << 40
    frame.release()
    for r in res[1:]:
        for k in r:
            assert gu.rel_err(r[k].cpu().numpy(), res[0][k].cpu().numpy()) <= 1e-6, k


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_adjoint_reaches_its_surfels_only(bad):
    """A non-finite colour adjoint at one pixel: every surfel blended there gets
    a non-finite colour gradient, and the surfels outside the pixel's tile get
    what they get without it."""
    from paper_2411_00771_gb300 import binding as B
    scene, cam, _, _ = syn.tiny_scene(seed=61, n=600, width=64, height=48, fx=60.0)
    sc, d, out, cnt, frame = gu.gpu_render(scene, cam)
    H, W = 48, 64
    rng = np.random.default_rng(4)
    adj = torch.from_numpy(rng.normal(size=(11, H, W)).astype(np.float32)).cuda()
    y, x = np.argwhere(cnt.cpu().numpy() >= 2)[0]
    res = []
    for v in (0.0, bad):
        a = adj.clone()
        a[0, y, x] = v
        g = {k: torch.zeros_like(t) for k, t in d.items()}
        sc.backward(frame, [a], [0x7], g)
        torch.cuda.synchronize()
        res.append(g["sh"].cpu().numpy()[:, 0, 0])
    one = np.zeros((1, 11, H, W))
    one[0, 0, y, x] = 1.0
    touched = oracle.backward(scene, cam, one)["sh"].reshape(600, -1)[:, 0] != 0
    assert touched.any() and not np.isfinite(res[1][touched]).any()
    vals, ranges, _ = frame.lists()
    lo, hi = ranges.cpu().numpy()[(y // 16) * ((W + 15) // 16) + x // 16]
    outside = np.ones(600, bool)
    outside[vals.cpu().numpy()[lo:hi]] = False
    assert np.array_equal(res[0][outside], res[1][outside])
