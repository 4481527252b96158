"""The update of K-means, exact for every binary16 input: the objective is the
sum of squared distances (an integer in units of 2^-48), the centroid the
rounded mean, at the edges of the kernel's steps, at every alignment of the
codebook and the SH rows and for values whose differences need more than 32 bits."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _fixed(h):
    """binary16 -> Python integers in units of 2^-24"""
    return (h.astype(np.float64) * 2.0 ** 24).astype(np.int64).astype(object)


@pytest.mark.parametrize("big", [False, True], ids=["usual", "large"])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("m", [1, 31, 32, 33, 2500])
def test_objective_and_centroids_are_exact(m, deg, offset, big):
    from paper_2411_00771_gb300 import binding as B
    C, K = 3 * (deg + 1) ** 2, 40  # K no multiple of 256: the FP32 assignment
    rng = np.random.default_rng(10 * m + deg)
    x = rng.normal(0.0, 0.3, (m, C))
    x[rng.random((m, C)) < 0.1] *= 1e-6  # subnormals
    if big:
        x[:, 0] = 150.0
        x[0, 0] = -150.0  # 300 apart: more than 2^32 units
    buf = torch.empty(m * C + offset, device="cuda")
    sh = buf[offset:].view(m, C // 3, 3)
    sh.copy_(torch.from_numpy(x.astype(np.float16).astype(np.float32).reshape(m, C // 3, 3)))
    keep = torch.zeros(m, dtype=torch.uint8, device="cuda")
    u = torch.from_numpy(rng.random(K).astype(np.float32)).cuda()
    xi = _fixed(x.astype(np.float16))

    def run(iters):
        buf = torch.empty(K * C + offset, dtype=torch.float16, device="cuda")
        cb = buf[offset:]
        assign = torch.empty(m, dtype=torch.int32, device="cuda")
        obj = torch.empty(iters + 1, dtype=torch.float64, device="cuda")
        got = ctypes.c_int64()
        B._check(B.lib().gs_vq_kmeans(m, deg, B._ptr(sh), B._ptr(keep, torch.uint8), K, iters, B._ptr(u),
                                      B._ptr(cb, torch.float16), B._ptr(assign, torch.int32),
                                      B._ptr(obj, torch.float64), 0, ctypes.byref(got), None))
        torch.cuda.synchronize()
        assert got.value == m
        return cb.view(K, C).cpu().numpy(), assign.cpu().numpy(), obj.cpu().numpy()

    c0, a0, o0 = run(0)
    exact = sum(int((d * d).sum()) for d in (xi - _fixed(c0)[a0])) * 2.0 ** -48
    # a sum of at most 2500 rounded terms, all positive
    assert abs(o0[0] - exact) <= 1e-12 * exact
    c1, _, o1 = run(1)
    assert abs(o1[0] - exact) <= 1e-12 * exact
    want = c0.copy()
    for j in range(K):
        mine = xi[a0 == j]
        if len(mine):
            s = np.array([int(v) for v in mine.sum(axis=0)], np.float64)
            want[j] = (s * 2.0 ** -24 / len(mine)).astype(np.float16)
    assert np.array_equal(c1.view(np.uint16), want.view(np.uint16))
