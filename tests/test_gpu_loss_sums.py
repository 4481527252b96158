"""The losses' sums over many tiles: tiles of large differences and, further
on, of small ones, whose sums FP32 would lose against the large.  Every
difference and every tile's sum is a binary fraction that FP32 holds, so the
losses are exact up to one rounding to FP32 (2^-24; four times that is
allowed)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

TW, TH = 32, 54  # the loss's tiles


def test_small_tiles_count_beside_large_ones():
    from paper_2411_00771_gb300 import binding as B
    gx, gy = 120, 40
    H, W = gy * TH, gx * TW
    d = np.zeros((3, H, W), np.float32)
    d[:, TH // 2::TH, TW // 2::TW] = 0.875
    for b in range(256):
        y, x = b // gx * TH, b % gx * TW
        d[0, y:y + TH, x:x + TW] = 16384.0
    out = torch.zeros((12, H, W), device="cuda")
    out[:3] = torch.from_numpy(d)
    out[5] = out[0]
    target, tinv = torch.zeros((3, H, W), device="cuda"), torch.zeros((H, W), device="cuda")
    losses, _, _, _ = B.loss(out, target, tinv, (0.8, 0.2, 0.5), adj_total=torch.zeros((11, H, W), device="cuda"))
    l1, _, depth, _ = [float(x) for x in losses.double().cpu()]
    for got, want in ((l1, d.astype(np.float64).mean()), (depth, d[0].astype(np.float64).mean())):
        assert abs(got - want) <= 2.0 ** -22 * want, got / want - 1
