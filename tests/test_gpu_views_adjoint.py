"""The several-view per-item adjoint orders a warp's Gaussians by their
numbers of views once a scene has enough of them (320,000 here): the
gradients of a small scene spread among Gaussians too faint to be seen equal
the small scene's own, for few views and for more than the 64 that one mask
holds, at a number of Gaussians that fills no whole warp.

Tolerance: the same addends in other orders of float32 atomics, N 2^-24 with
at most a few thousand addends per entry but signs that cancel: 1e-4 of the
group's norm; the faint Gaussians' gradients are exactly 0.
"""
import numpy as np
import pytest
import torch

from paper_2311_18561_gb300 import render as R
from paper_2311_18561_gb300 import synth

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("degree", [0, 3])
@pytest.mark.parametrize("n_views", [3, 66])
def test_gradients_among_unseen_gaussians(n_views, degree):
    few, many = 1500, 320_021
    scene = synth.make_plain_scene(seed=6, n=few, sh_degree=degree)
    at = np.sort(np.random.default_rng(2).choice(many, few, replace=False))
    wide = {}
    for k, v in scene.items():
        wide[k] = np.repeat(v[:1], many, axis=0)
        if k == "opacity":
            wide[k][:] = 1e-4
        wide[k][at] = v
    # the views look at different parts, so the numbers of views differ
    cams = [synth.plain_camera(80 + v % 3, 60, t=0.3 + 0.01 * v) for v in range(n_views)]
    for v, c in enumerate(cams):
        c["cx"] += 40.0 * (v % 3 - 1)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    d = [dict(rgb=torch.randn(3, c["height"], c["width"], generator=g, device="cuda")) for c in cams]
    grads = []
    for s in (scene, wide):
        r, fr, st = R.Renderer(), R.Frame(), R.scene_to_device(s)
        r.forward(st, cams, frame=fr)
        grads.append(r.backward(st, cams, fr, d))
        r.close()
        fr.close()
    where = torch.tensor(at, device="cuda")
    faint = torch.ones(many, dtype=torch.bool, device="cuda")
    faint[where] = False
    for k in R.PARAM_NAMES:
        a, b = grads[0][k], grads[1][k][where]
        assert torch.linalg.norm(a) > 0, k
        assert torch.linalg.norm((a - b).double()) <= 1e-4 * torch.linalg.norm(a.double()), k
        assert not grads[1][k][faint].any(), k
