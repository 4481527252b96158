"""What a kept frame holds on the device: per surfel the blend record,
footprint, rectangle, tile count and candidate index, per pixel the two
positions of the backward, per tile its range and place, and per instance the
surfel (4 bytes) and the block mask (2 bytes)."""
import ctypes

import pytest
import torch

from paper_2411_00771_gb300 import synthetic as syn
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,W,H", [(3000, 96, 80), (20_000, 200, 150), (50, 16, 16)])
def test_kept_frame_bytes(n, W, H):
    from paper_2411_00771_gb300 import binding as B
    scene, cam, _, _ = syn.tiny_scene(seed=n, n=n, width=W, height=H, fx=float(W))
    d = gu.to_dev(scene)
    live = {}

    def alloc(size, ctx, stream):
        t = torch.empty(size, dtype=torch.uint8, device="cuda")
        live[t.data_ptr()] = t
        return t.data_ptr()

    def free(ptr, size, ctx, stream):
        torch.cuda.synchronize()
        live.pop(ptr)

    names = ("mu", "quat", "scale", "opacity", "sh")
    desc = B.gs_scene_desc()
    desc.settings, desc.sh_degree = B.default_settings(), scene["sh_degree"]
    desc.allocator = B.gs_allocator(B.ALLOC_FN(alloc), B.FREE_FN(free), None)
    sc = B.Scene(*[d[k] for k in names], scene["sh_degree"])
    B._check(B.lib().gs_destroy_scene(sc._handle))
    sc._handle = ctypes.c_void_p()
    sc._fill(desc, *[d[k] for k in names])
    B._check(B.lib().gs_create_scene(ctypes.byref(sc._handle), ctypes.byref(desc)))
    sc._keep = desc
    out, frame = sc.render(cam)
    torch.cuda.synchronize()
    K = frame.lists()[0].numel()
    tiles = ((W + 15) // 16) * ((H + 15) // 16)
    held = sum(t.numel() for t in live.values())
    assert K > 0 and held == n * (112 + 56 + 8 + 4 + 4) + W * H * 8 + tiles * 12 + 64 + K * 6
    frame.release()
    torch.cuda.synchronize()
    assert not live
    again, _ = sc.render(cam, save=False)
    assert torch.equal(again, out) and not live
