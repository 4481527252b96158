"""The backward under a memory limit: at most sixteen replays, then out of
memory, with nothing done.  The parts' gradients within 1e-4 of the whole's, a
tenth of the gate against the oracle: they are the same FP32 sums in another
order."""
import numpy as np
import pytest
import torch

from paper_2411_00771_gb300 import synthetic as syn
from tests import gpu_util as gu
from tests.test_gpu_blend_edges import LOSS, _limited_scene

pytestmark = pytest.mark.gpu

N = 3000
RECORD = 64  # bytes per surfel


@pytest.mark.parametrize("masks", [LOSS, [0x7FF]], ids=["loss", "all"])
def test_backward_refuses_below_a_sixteenth(masks):
    from paper_2411_00771_gb300 import binding as B
    scene, cam, _, _ = syn.tiny_scene(seed=56, n=N, width=48, height=40, fx=45.0)
    d = gu.to_dev(scene)
    limit = [1 << 40]
    sc, sizes = _limited_scene(d, scene["sh_degree"], limit)
    out, frame = sc.render(cam)
    adj = [torch.from_numpy(np.random.default_rng(7).normal(size=(11, 40, 48)).astype(np.float32)).cuda()
           for _ in masks]

    def backward():
        g = {k: torch.zeros_like(v) for k, v in d.items()}
        screen = torch.zeros((len(masks), N, 2), device="cuda")
        sc.backward(frame, adj, masks, g, screen)
        torch.cuda.synchronize()
        return {**g, "screen": screen}

    full = backward()
    part = -(-N // 16) * RECORD
    limit[0] = part
    again = backward()
    assert sizes[-1] == part
    for k in full:
        assert gu.rel_err(again[k].cpu().numpy(), full[k].cpu().numpy()) <= 1e-4, k
    count = len(sizes)
    limit[0] = part - 1
    g = {k: torch.zeros_like(v) for k, v in d.items()}
    with pytest.raises(B.GsError) as e:
        sc.backward(frame, adj, masks, g)
    assert e.value.code == -2
    torch.cuda.synchronize()
    assert len(sizes) == count and all(not bool(v.any()) for v in g.values())
    limit[0] = 1 << 40
    frame.release()
