"""The loss where the image ends on and beside its tiles (32 x 54) and for
buffers that start inside an allocation, against the FP64 oracle at the
tolerances of the parity tests."""
import numpy as np
import pytest
import torch

import oracle
from tests.test_gpu_parity import _synthetic_render_planes

pytestmark = pytest.mark.gpu


def _dev(a, offset):
    buf = torch.empty(a.size + offset, device="cuda")
    buf[offset:] = torch.from_numpy(a.ravel())
    return buf[offset:].view(a.shape)


@pytest.mark.parametrize("depth", [True, False])
@pytest.mark.parametrize("W,H", [(1, 1), (40, 1), (3, 120), (31, 53), (32, 54), (33, 55), (64, 108), (65, 109), (97, 49)])
def test_loss_at_the_edges_of_tiles(W, H, depth):
    from paper_2411_00771_gb300 import binding as B
    rng = np.random.default_rng(W * 1000 + H)
    out = _synthetic_render_planes(rng, H, W).astype(np.float32)
    tgt = rng.uniform(0, 1, (3, H, W)).astype(np.float32)
    tinv = rng.uniform(0.1, 0.6, (H, W)).astype(np.float32) if depth else None
    w = (0.8, 0.2, 0.5 if depth else 0.0)
    ref = oracle.loss(out, tgt, tinv, w)
    offset = (W + H) % 4
    adj = [torch.zeros((11, H, W), device="cuda") for _ in range(3)]
    losses, _, _, _ = B.loss(_dev(out, offset), _dev(tgt, offset), None if tinv is None else _dev(tinv, offset), w,
                             adj_total=adj[0], adj_ssim=adj[1], adj_l1=adj[2])
    l = losses.cpu().numpy()
    assert abs(l[0] - ref["l1"]) < 1e-6 and abs(l[1] - ref["ssim"]) < 1e-5
    assert abs(l[2] - ref["depth"]) < 1e-6 and abs(l[3] - ref["total"]) < 1e-5
    for got, exp in zip(adj, ref["adj"]):
        assert np.abs(got.cpu().numpy() - exp).max() <= 1e-4 * max(np.abs(exp).max(), 1e-30)
