"""A pixel that does not blend an entry has the weight zero, which must only
ever meet finite values: values and output gradients that are each finite but
whose product is not, and the sums of a pixel that an infinite value has
reached, stay with the Gaussians blended at the pixels that see that value.
All others keep the gradients they have without it (equal sums in another
order: 1e-4 of the norm).
"""
import numpy as np
import pytest
import torch

from paper_2311_18561_gb300 import abi
from paper_2311_18561_gb300 import render as R
from paper_2311_18561_gb300 import synth

from .test_gpu_warp_blocks import _views

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

N, CAM = 300, synth.plain_camera(75, 53, t=0.5)


@pytest.mark.parametrize("repeat", [False, True])  # two pixels per lane, and four or eight
@pytest.mark.parametrize("cfg", [(8, 8, 1), (16, 16, 1), (32, 32, 4)])
@pytest.mark.parametrize("what", ["colour", "channel", "infinite colour", "infinite channel"])
def test_zero_weights_meet_finite_values_only(what, cfg, repeat):
    scene = synth.make_plain_scene(seed=9, n=N, log_scale_mean=-3.0)
    st = R.scene_to_device(scene)
    cams = _views(CAM, cfg) if repeat else [CAM]
    r, fr = R.Renderer(tile=cfg[:2], pixels_per_thread=cfg[2]), R.Frame()
    who = int(np.argmax(scene["opacity"]))
    # the pixels that see `who`, and the Gaussians blended there
    st["sem"] = torch.zeros(N, 1, device="cuda")
    st["sem"][who] = 1.0
    support = (r.forward(st, [CAM], features=abi.FEAT_SEM)[0]["feat"] > 0).float()
    st["sem"][:] = 1.0
    r.forward(st, [CAM], frame=fr, features=abi.FEAT_SEM)
    reached = r.backward(st, [CAM], fr, [dict(feat=support)])["sem"][:, 0] > 0
    assert 0 < int(reached.sum()) < N
    huge = "infinite" not in what  # finite alone, their product not
    features = abi.FEAT_SEM if "channel" in what else 0
    name = "feat" if features else "rgb"
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    dl = torch.randn(1 if features else 3, CAM["height"], CAM["width"], generator=g, device="cuda").abs() + 0.5
    if huge:
        dl *= 5e13
    value = 1e25 if huge else float("inf")
    grads = []
    for v in (0.25, value):
        if features:
            st["sem"][who] = v
        else:
            st["sh"][who] = 0.0
            st["sh"][who, 0] = v / 0.28
        r.forward(st, cams, frame=fr, features=features)
        grads.append(r.backward(st, cams, fr, [{name: dl}] * len(cams)))
    assert not torch.isfinite(grads[1]["opacity"][reached]).all()
    for k in ("mu", "scale", "quat", "opacity"):
        want, got = (x[k].reshape(N, -1)[~reached] for x in grads)
        assert torch.isfinite(want).all()
        assert torch.isfinite(got).all(), (k, int((~torch.isfinite(got)).any(1).sum()))
        assert torch.linalg.norm(want) > 0
        assert torch.linalg.norm(got - want) <= 1e-4 * torch.linalg.norm(want), k
