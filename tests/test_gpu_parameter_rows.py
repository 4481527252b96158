"""The preprocess moves SH rows by 16-byte pieces, by words or lane by lane, as
degree, storage and alignment allow, and reads quaternions and scales whole
where they are aligned.  The values read are the same, so a render is the same
bits for every storage of the same parameters, also where the surfels end
inside a warp or a block."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_00771_gb300 import binding as B
from paper_2411_00771_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def _shifted(t, elements):
    """A contiguous copy of t that starts `elements` into its own buffer."""
    buf = torch.empty(t.numel() + elements, dtype=t.dtype, device=t.device)
    buf[elements:] = t.reshape(-1)
    return buf[elements:].view(t.shape)


def _image(sc, cam):
    out, frame = sc.render(cam)
    torch.cuda.synchronize()
    assert int((out[3] > 0).sum()) > 0
    frame.release()
    return out


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 1000])
def test_same_bits_for_every_storage(n, deg):
    scene, cam, _, _ = syn.tiny_scene(seed=40 + n, n=n, width=65, height=47, fx=60.0, sh_degree=deg, xy_range=0.3)
    keys = ("mu", "quat", "scale", "opacity", "sh")
    p = {k: torch.from_numpy(np.float32(oracle.half(np.asarray(scene[k], np.float64)))).cuda() for k in keys}
    p["mu"] = torch.from_numpy(np.ascontiguousarray(scene["mu"], np.float32)).cuda()
    ref = _image(B.Scene(*[p[k] for k in keys], deg), cam)
    for s in (1, 2, 3):
        q = {k: _shifted(v, s) for k, v in p.items()}
        assert torch.equal(_image(B.Scene(*[q[k] for k in keys], deg), cam), ref), s
    C = 3 * (deg + 1) ** 2
    table = p["sh"].reshape(n, C).half()
    comp = {"mu": p["mu"], "quat": p["quat"].half(), "scale": p["scale"].half(), "opacity": p["opacity"].half(),
            "sh_row": torch.arange(n - 1, -1, -1, dtype=torch.int32, device="cuda"), "sh_degree": deg}
    for s in (0, 1, 4):
        comp["sh_table"] = _shifted(table.flip(0).contiguous(), s)
        assert torch.equal(_image(B.CompressedScene(comp), cam), ref), ("half", s)
