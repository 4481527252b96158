"""Block masks made at emission and carried in the sort's keys (images of up to
65536 tiles) against masks made per sorted instance (larger images): the same
camera with a larger image gives the same bits in the part both have."""
import numpy as np
import pytest
import torch

from paper_2411_00771_gb300 import synthetic as syn
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scales", [(-9.0, -7.0), (-7.0, -3.5)], ids=["dots", "wide"])
@pytest.mark.parametrize("W,H,n", [(4352, 4096, 20000), (4096, 4352, 20000), (4097, 4096, 33)])
def test_masks_in_keys_and_per_instance_agree(W, H, n, scales):
    w, h = min(W, 4096), min(H, 4096)  # at most 65536 tiles
    scene, cam, _, _ = syn.tiny_scene(seed=W + n, n=n, width=w, height=h, fx=2200.0, log_scale_range=scales)
    _, _, small, cs, _ = gu.gpu_render(scene, dict(cam, width=w, height=h))
    _, _, large, cl, _ = gu.gpu_render(scene, dict(cam, width=W, height=H))
    # footprints that the smaller image's edge cuts have a smaller rectangle
    # (and with it another grid of their offsets): a margin is left out
    mx, my = (w if W == w else 3000), (h if H == h else h - 1000)
    assert int((cs[:my, :mx] > 0).sum()) > 0
    assert torch.equal(cs[:my, :mx], cl[:my, :mx])
    assert torch.equal(small[:, :my, :mx], large[:, :my, :mx])


@pytest.mark.parametrize("scales", [(-13.0, -11.0), (-11.0, -8.5)], ids=["dots", "wide"])
def test_rows_of_many_tiles(scales):
    """16384 tiles in a row take the masks in the keys, 16385 do not."""
    scene, cam, _, _ = syn.tiny_scene(seed=8, n=20000, width=16384 * 16, height=16, fx=2.0e5, log_scale_range=scales)
    scene["mu"][:, 1] *= 2e-5
    _, _, small, cs, _ = gu.gpu_render(scene, cam)
    _, _, large, cl, _ = gu.gpu_render(scene, dict(cam, width=16385 * 16))
    mx = 16384 * 16 - 1000
    assert int((cs[:, 66000:mx] > 0).sum()) > 0
    assert torch.equal(cs[:, :mx], cl[:, :mx])
    assert torch.equal(small[:, :, :mx], large[:, :, :mx])
