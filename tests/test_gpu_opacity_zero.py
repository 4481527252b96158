"""Opacity gradients of surfels of no or hardly any opacity, which blend where
alpha_min is 0: d alpha / d opacity = exp(-rho / 2) does not vanish with the
opacity.  Against the FP64 oracle at the parity tests' gate (1e-3)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_00771_gb300 import synthetic as syn
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

FLAGS = oracle.FLAG_RHO | oracle.FLAG_TSTOP | oracle.FLAG_MEDIAN | oracle.FLAG_BRANCH


@pytest.mark.parametrize("masks", [[0x7 | (1 << 5), 0x7, 0x7], [0x7FF]], ids=["loss", "all"])
def test_opacity_gradient_without_opacity(masks):
    scene, cam, _, _ = syn.tiny_scene(seed=71, n=600, width=64, height=48, fx=60.0)
    scene["opacity"] = scene["opacity"].copy()
    scene["opacity"][0::4] = 0.0
    scene["opacity"][1::4] = 1e-30
    settings = dict(alpha_min=0.0)
    sc, d, out, cnt, frame = gu.gpu_render(scene, cam, settings)
    ref = oracle.render(scene, cam, settings=settings)
    ok = (ref["flags"] & FLAGS) == 0
    assert ok.mean() > 0.5
    rng = np.random.default_rng(5)
    adj = rng.normal(size=(len(masks), 11, 48, 64)) * ok
    for s, m in enumerate(masks):
        for p in range(11):
            if not (m >> p) & 1:
                adj[s, p] = 0.0
    adj = np.float32(adj)
    grads = {k: torch.zeros_like(x) for k, x in d.items()}
    sc.backward(frame, [torch.from_numpy(a).cuda() for a in adj], masks, grads)
    torch.cuda.synchronize()
    want = oracle.backward(scene, cam, adj.astype(np.float64), settings=settings)["opacity"].ravel()
    got = grads["opacity"].cpu().numpy().ravel()
    for part in (slice(0, None, 4), slice(1, None, 4), slice(2, None, 2)):
        assert np.abs(want[part]).max() > 0
        assert gu.rel_err(got[part], want[part]) <= 1e-3
