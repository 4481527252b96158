"""Long lists composited in segments: lists that end on and beside a segment's
end, pixels that stop in the first segment, in a later one and never, side by
side in a tile, and images that end inside it.  Against the FP64 oracle at the
tolerances of the parity tests."""
import numpy as np
import pytest

from paper_2411_00771_gb300 import synthetic as syn
from tests import test_gpu_blend_edges as be

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["faint", "opaque", "mixed"])
@pytest.mark.parametrize("W,H,n", [(16, 16, 1025), (16, 16, 2048), (16, 16, 2049), (13, 9, 3100), (21, 19, 1300)])
def test_segments(W, H, n, kind):
    rng = np.random.default_rng(n + W)
    q = rng.normal(0.0, 0.05, (n, 4))
    q[:, 0] = 1.0
    mu = np.column_stack([rng.uniform(-0.05, 0.05, (n, 2)), rng.uniform(2, 4, n)])
    scale = rng.uniform(1.0, 1.5, (n, 2))
    opacity = rng.uniform(0.0045, 0.006, n)  # about e^-9 after 2000: some pixels stop late, some never
    if kind == "opaque":
        opacity = rng.uniform(0.05, 0.6, n)
    if kind == "mixed":  # small opaque disks over a part of the image, among the faint wide ones
        k = rng.random(n) < 0.3
        mu[k, 0] = rng.uniform(-0.8, 0.0, k.sum())
        scale[k] = rng.uniform(0.05, 0.2, (k.sum(), 2))
        opacity[k] = rng.uniform(0.2, 0.9, k.sum())
    scene = dict(mu=mu.astype(np.float32), quat=q.astype(np.float32), scale=scale.astype(np.float32),
                 opacity=opacity.astype(np.float32), sh=rng.normal(0, 0.5, (n, 1, 3)).astype(np.float32), sh_degree=0)
    be._check(scene, syn.identity_camera(W, H, float(W)), be.LOSS, seed=n)
