"""Scans and sorts of few items by one block: lists and ranges bit for bit
where the surfels or the instances end on and beside the sizes at which the
route changes, with equal depths (the order of ties is by index)."""
import numpy as np
import pytest

from paper_2411_00771_gb300 import synthetic as syn
from tests import gpu_util as gu
from tests import rowrule as rr

pytestmark = pytest.mark.gpu

RF = np.float32(np.sqrt(9.0 / 2.0))


@pytest.mark.parametrize("W,H", [(16, 16), (64, 48), (1500, 900)], ids=["one_tile", "few_tiles", "many_tiles"])
@pytest.mark.parametrize("n", [1, 2, 33, 1023, 4095, 4096, 4097, 16383, 16384, 16385])
def test_lists_beside_the_route_changes(n, W, H):
    # dots of less than a pixel and the filter's two: about one to three tiles each
    scene, cam, _, _ = syn.tiny_scene(seed=n, n=n, width=W, height=H, fx=0.6 * W, xy_range=0.8,
                                      log_scale_range=(-9.0, -8.0))
    scene["mu"][::3, 2] = 2.5  # ties
    sc, d, out, cnt, frame = gu.gpu_render(scene, cam)
    vals, ranges, _ = [t.cpu().numpy() for t in frame.lists()]
    geom, depth, tcount = [t.cpu().numpy() for t in frame.cover()]
    frame.release()
    tiles_x, tiles_y = (W + 15) // 16, (H + 15) // 16
    surf, tile = rr.instances(geom, np.nonzero(tcount > 0)[0], tiles_x, RF)
    exp_vals, exp_ranges = rr.sorted_lists(surf, tile, depth.view(np.uint32), tiles_x * tiles_y)
    assert len(exp_vals) > 0 or n <= 2
    assert np.array_equal(vals, exp_vals)
    assert np.array_equal(ranges, exp_ranges)
