"""Trim contribution of faint disks that cover a whole 4K view: half a million
4 x 4 blocks add nearly the same value to one sum.  Against the FP64 oracle at
the contribution tests' tolerance (1e-5 relative); the support and every
threshold are far away, so nothing is uncertain."""
import numpy as np
import pytest

import oracle
from paper_2411_00771_gb300 import synthetic as syn
from tests.test_gpu_contribution import SUM_ATOL, SUM_RTOL, _gpu_view

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma", [0.5, 1.0, 0.0])
def test_wide_faint_disks(gamma):
    n = 4
    scene = dict(mu=np.float32([[0.1, -0.1, 3.0], [0.0, 0.2, 3.1], [-0.2, 0.0, 3.2], [0.1, 0.1, 3.3]]),
                 quat=np.float32([[1, 0, 0, 0]] * n), scale=np.float32([[200, 190], [210, 180], [220, 205], [195, 200]]),
                 opacity=np.float32([0.013, 0.021, 0.017, 0.011]), sh=np.zeros((n, 1, 3), np.float32), sh_degree=0)
    cam = syn.identity_camera(3840, 2160, 3840.0)
    ref = oracle.contribution(scene, cam, gamma=gamma)
    assert np.all(ref["flag_sum"] == 0) and np.all(ref["count"] == 3840 * 2160)
    s, c = _gpu_view(scene, cam, gamma)
    assert np.array_equal(c, ref["count"])
    assert np.all(np.abs(s - ref["sum"]) <= SUM_ATOL + SUM_RTOL * ref["sum"]), np.abs(s / ref["sum"] - 1).max()
