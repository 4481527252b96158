"""The visibility count decides most pairs by clear-cut tests and the rest by
the definition, and shares the views of few points out over blocks.  A near
plane of 1e-3 or less takes the definition throughout, so with no point between
the two near planes used here both give the same counts, whatever the views,
sizes and settings."""
import numpy as np
import pytest
import torch

from paper_2411_00771_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def _views(rng, k):
    out = []
    for i in range(k):
        W, H = [(320, 180), (64, 640), (1, 1), (1920, 1080), (37, 53)][i % 5]
        c = dict(syn.orbit_camera(rng, W, H, radius=rng.uniform(30, 140), altitude=rng.uniform(5, 90)))
        if i % 3 == 1:  # principal point outside the image, focal lengths apart
            c.update(cx=c["cx"] + 2.0 * W, fy=0.3 * c["fy"])
        if i % 7 == 3:  # lenses out of the ordinary
            c.update(fx=c["fx"] * 1e5, fy=c["fy"] * 1e-6)
        out.append(c)
    return out


@pytest.mark.parametrize("sigma,lowpass", [(0.0, 0.0), (0.2, 0.3), (30.0, 0.0), (1e-3, 400.0)])
@pytest.mark.parametrize("n,k", [(1, 1), (511, 15), (512, 16), (513, 17), (2000, 128), (2000, 129), (700_000, 40)])
def test_same_counts_as_the_definition(n, k, sigma, lowpass):
    from paper_2411_00771_gb300 import binding as B
    rng = np.random.default_rng(n + k)
    cams = _views(rng, k)
    pts = rng.uniform([-120, -120, -5], [120, 120, 60], (n, 3)).astype(np.float32)
    pts[::97] *= 1e4
    pts[::1013] *= 1e30
    pts[50::2003] = np.nan
    pts[70::2011, 1] = np.inf
    # no point between the two near planes in any view
    R = np.array([np.asarray(c["R"], np.float32).reshape(3, 3)[2] for c in cams])
    t = np.array([np.float32(c["t"][2]) for c in cams])
    with np.errstate(all="ignore"):
        z = pts.astype(np.float64) @ R.T.astype(np.float64) + t
    pts = pts[~((z > -0.01) & (z < 0.01)).any(axis=1)]
    d = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
    fast = B.visibility_count(d, sigma, cams, near_plane=0.0011, lowpass=lowpass)
    slow = B.visibility_count(d, sigma, cams, near_plane=0.001, lowpass=lowpass)
    assert torch.equal(fast, slow)
    B.visibility_count(d, sigma, cams, counts=fast, near_plane=0.0011, lowpass=lowpass)  # accumulates
    assert torch.equal(fast, 2 * slow)
