"""The render and its gradients, bit for bit.

The FP32 sums of a long disk seen nearly edge-on cancel, so that its gradients
follow the rounding of every term and the order of every addition.  The golden
values were computed by the kernels as they were before the blends were split
into lane groups, and pin the terms and the order within a warp: every surfel
lies within one 8 x 8 pixel block, so that one warp makes its sums and no order
of atomic additions plays a part.  Scene and adjoints are made of small
fractions, the same on every machine."""
import os

import numpy as np
import pytest
import torch

from paper_2411_00771_gb300 import synthetic as syn
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "backward_order.npz")
W, H, FX, PER_BLOCK = 64, 48, 60.0, 6
MASKS = {"loss": [0x7 | (1 << 5), 0x7, 0x7], "all": [0x7FF], "all3": [0x7FF, 0x7, 0x7]}


def _frac(i, p, q):
    """Values in [-1, 1) that look random: i p mod q over q, in 64-bit integers."""
    return ((i * p) % q).astype(np.float64) / q * 2 - 1


def scene():
    n = (W // 8) * (H // 8) * PER_BLOCK
    i = np.arange(n, dtype=np.int64) + 1
    block = (i - 1) // PER_BLOCK
    z = 3.0 + 0.9 * _frac(i, 7919, 1009)
    px = 8.0 * (block % (W // 8)) + 4.0 + 0.8 * _frac(i, 104729, 2003)
    py = 8.0 * (block // (W // 8)) + 4.0 + 0.8 * _frac(i, 15485863, 3001)
    mu = np.stack([(px - W / 2) * z / FX, (py - H / 2) * z / FX, z], 1)
    quat = np.stack([_frac(i, 31, 4001), _frac(i, 1237, 5003), _frac(i, 99991, 6007), _frac(i, 65537, 7001) + 0.01], 1)
    # half-axes of 0.1 to 1 pixels: three of them end within the block
    scale = np.stack([0.55 + 0.4 * _frac(i, 271, 997), 0.55 + 0.45 * _frac(i, 613, 991)], 1) * z[:, None] / FX
    sh = np.stack([_frac(i, 11 + k, 8009) for k in range(12)], 1).reshape(n, 4, 3)
    return dict(mu=np.float32(mu), quat=np.float32(quat), scale=np.float32(scale),
                opacity=np.float32(0.55 + 0.44 * _frac(i, 43, 1021)), sh=np.float32(sh), sh_degree=1)


def gradients(masks):
    sc, d, out, cnt, frame = gu.gpu_render(scene(), syn.identity_camera(W, H, FX))
    k = np.arange(len(masks) * 11 * H * W, dtype=np.int64) + 1
    adj = np.float32(_frac(k, 7368787, 100003)).reshape(len(masks), 11, H, W)
    n = d["mu"].shape[0]
    grads = {k: torch.zeros_like(x) for k, x in d.items()}
    screen = torch.zeros((len(masks), n, 2), device="cuda")
    sc.backward(frame, [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in adj], masks, grads, screen)
    torch.cuda.synchronize()
    frame.release()
    return {"out": out.cpu().numpy(), "screen": screen.cpu().numpy(), **{k: v.cpu().numpy() for k, v in grads.items()}}


@pytest.mark.parametrize("name", list(MASKS))
def test_gradients_are_the_golden_ones(name):
    got = gradients(MASKS[name])
    golden = np.load(GOLDEN)
    for k, v in got.items():
        want = golden["out" if k == "out" else name + "/" + k]
        assert np.array_equal(v, want), k
