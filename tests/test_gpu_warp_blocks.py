"""The compositing kernels' pixel blocks: a frame small enough for two pixels
per lane and the same view repeated until a lane takes four (forward) and
eight (adjoint) give the same images bit for bit and gradients that add up,
at ragged sizes and for every tile shape; non-finite colours and output
gradients stay with the pixels and Gaussians that blend them.

Tolerance of the summed gradients: equal addends, so N times the single
view's gradient up to the rounding of N float32 additions (N 2^-24 = 1.8e-5
at 300 views) and of the two kernels' different summation orders (below 1e-5
in norm): 1e-4 of the group's norm.
"""
import numpy as np
import pytest
import torch

from paper_2311_18561_gb300 import abi
from paper_2311_18561_gb300 import render as R
from paper_2311_18561_gb300 import synth
from paper_2311_18561_gb300 import tune as T

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def _views(cam, cfg):
    """Copies of cam whose tiles are 66 blocks of 256 pixels per SM together."""
    tx, ty = R.tiles_of(cam, cfg[:2])
    return [cam] * (66 * R.device_sm_count() * 256 // (tx * ty * cfg[0] * cfg[1]) + 1)


def _weights(cam, aux, seed=5):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    h, w = cam["height"], cam["width"]
    d = dict(rgb=torch.randn(3, h, w, generator=g, device="cuda"))
    if aux:
        d["depth"] = torch.randn(h, w, generator=g, device="cuda")
        d["alpha"] = torch.randn(h, w, generator=g, device="cuda")
    return d


@pytest.mark.parametrize("aux", [False, True])
@pytest.mark.parametrize("cfg", T.CONFIGS)
def test_blocks_of_every_width_agree(cfg, aux):
    scene = synth.make_plain_scene(seed=4, n=300, sh_degree=1, log_scale_mean=-2.3)
    scene["opacity"][::7] = 1.0  # alphas at the cap
    st = R.scene_to_device(scene)
    cam = synth.plain_camera(97, 61, t=0.4, bg=(0.2, 0.1, 0.3))
    r = R.Renderer(tile=cfg[:2], pixels_per_thread=cfg[2])
    d = _weights(cam, aux)
    one, many = R.Frame(), R.Frame()
    ref = r.forward(st, [cam], frame=one)[0]
    g1 = r.backward(st, [cam], one, [d])
    cams = _views(cam, cfg)
    outs = r.forward(st, cams, frame=many)
    gn = r.backward(st, cams, many, [d] * len(cams))
    for v in (0, len(cams) // 2, len(cams) - 1):
        for k in ("rgb", "depth", "alpha"):
            assert torch.equal(outs[v][k], ref[k]), (v, k)
    for k in R.PARAM_NAMES:
        want = g1[k].double() * len(cams)
        assert torch.linalg.norm(want) > 0, k
        assert torch.linalg.norm(gn[k].double() - want) <= 1e-4 * torch.linalg.norm(want), k


@pytest.mark.parametrize("size", [(97, 61), (161, 37)])
@pytest.mark.parametrize("cfg", T.CONFIGS)
def test_one_and_two_pixels_per_lane_agree(cfg, size):
    """The compositor's pixels per lane in a small frame follow from the
    number of items per block of pixels: Gaussians too faint to be seen take
    the same view through one pixel per lane (36 items per block) and two
    (about 5 and 300), with the same images bit for bit, gradients that agree
    (equal sums in another order: 1e-4 of the norm) and infinite colours in
    the same pixels."""
    scene = synth.make_plain_scene(seed=4, n=300, sh_degree=1, log_scale_mean=-2.3)
    scene["opacity"][::7] = 1.0
    cam = synth.plain_camera(*size, t=0.4, bg=(0.2, 0.1, 0.3))
    tx, ty = R.tiles_of(cam, cfg[:2])
    blocks = tx * ty * cfg[0] * cfg[1] / 128
    r = R.Renderer(tile=cfg[:2], pixels_per_thread=cfg[2])
    d = _weights(cam, True)
    for bad in (False, True):
        if bad:
            scene["sh"][int(np.argmax(scene["opacity"]))] = np.inf
        ref = None
        for per_block in (3, 36, 300):
            n = max(300, int(per_block * blocks)) - 300
            part = {k: np.concatenate([v, np.repeat(v[:1], n, axis=0)]) for k, v in scene.items()}
            part["opacity"][300:] = 1e-4
            fr = R.Frame()
            st = R.scene_to_device(part)
            out = r.forward(st, [cam], frame=fr)[0]
            cur = [out[k].clone() for k in ("rgb", "depth", "alpha")]
            if not bad:
                cur.append(r.backward(st, [cam], fr, [d])["opacity"][:300].clone())
            if ref is None:
                ref = cur
            for x, y in zip(ref[:3], cur[:3]):
                assert torch.equal(torch.nan_to_num(x, nan=7.0), torch.nan_to_num(y, nan=7.0)), (bad, per_block)
            for x, y in zip(ref[3:], cur[3:]):
                assert torch.linalg.norm(x - y) <= 1e-4 * torch.linalg.norm(x), per_block


@pytest.mark.parametrize("repeat", [False, True])
@pytest.mark.parametrize("cfg", [(16, 16, 1), (16, 8, 1), (32, 32, 4)])
def test_non_finite_values_stay_where_they_blend(cfg, repeat):
    scene = synth.make_plain_scene(seed=9, n=200, log_scale_mean=-2.3)
    st = R.scene_to_device(scene)
    cam = synth.plain_camera(75, 53, t=0.5)
    cams = _views(cam, cfg) if repeat else [cam]
    r = R.Renderer(tile=cfg[:2], pixels_per_thread=cfg[2])
    fr = R.Frame()
    # an infinite colour shows exactly where its Gaussian has a weight
    who = int(np.argmax(scene["opacity"]))
    st["sem"] = torch.zeros(200, 1, device="cuda")
    st["sem"][who] = 1.0
    weight = r.forward(st, [cam], features=abi.FEAT_SEM)[0]["feat"][0]
    bad = dict(st, sh=st["sh"].clone())
    bad["sh"][who] = float("inf")
    out = r.forward(bad, cams)[-1]
    assert 0 < int((weight > 0).sum()) < weight.numel()
    for c in range(3):
        assert torch.equal(~torch.isfinite(out["rgb"][c]), weight > 0)
    assert torch.isfinite(out["depth"]).all() and torch.isfinite(out["alpha"]).all()
    # a NaN output gradient reaches exactly the Gaussians its pixel blends
    y, x = (int(v) for v in np.argwhere((weight > 0).cpu().numpy())[0])
    st["sem"][:] = 1.0
    r.forward(st, [cam], frame=fr, features=abi.FEAT_SEM)
    pick = torch.zeros(1, 53, 75, device="cuda")
    pick[0, y, x] = 1.0
    blended = r.backward(st, [cam], fr, [dict(feat=pick)])["sem"][:, 0] > 0
    r.forward(st, cams, frame=fr)
    d = _weights(cam, False)
    d["rgb"][:, y, x] = float("nan")
    grads = r.backward(st, cams, fr, [d] * len(cams))
    assert 0 < int(blended.sum()) < 200
    assert torch.equal(~torch.isfinite(grads["opacity"]), blended)


@pytest.mark.parametrize("mask,n_sem", [(abi.FEAT_RHO, 0), (abi.FEAT_VBAR, 0), (abi.FEAT_SEM, 1), (abi.FEAT_SEM, 32),
                                        (abi.FEAT_VBAR | abi.FEAT_SEM, 30), (7, 19), (7, 32)])
def test_channels_keep_the_colour_pass_and_their_non_finite_values(mask, n_sem):
    """Colour, depth and opacity rendered with channels equal the plain
    render's bit for bit and their gradients agree (one view, equal sums in
    another order: 1e-4 of the norm); a class value that is not finite shows
    exactly where its Gaussian has a weight."""
    scene = synth.make_plain_scene(seed=9, n=200, log_scale_mean=-2.3)
    st = R.scene_to_device(scene)
    cam = synth.plain_camera(75, 53, t=0.5)
    r, fr, fp = R.Renderer(), R.Frame(), R.Frame()
    plain = r.forward(st, [cam], frame=fp)[0]
    if n_sem:
        st["sem"] = torch.tensor(synth.make_semantics(200, n_sem), device="cuda")
    out = r.forward(st, [cam], frame=fr, features=mask)[0]
    for k in ("rgb", "depth", "alpha"):
        assert torch.equal(out[k], plain[k]), k
    d = _weights(cam, True)
    want = r.backward(st, [cam], fp, [d])
    got = r.backward(st, [cam], fr, [dict(d, feat=torch.zeros_like(out["feat"]))])
    for k in R.PARAM_NAMES:
        assert torch.linalg.norm(got[k] - want[k]) <= 1e-4 * torch.linalg.norm(want[k]), k
    if n_sem:
        who = int(np.argmax(scene["opacity"]))
        st["sem"] = torch.zeros(200, n_sem, device="cuda")
        st["sem"][who, n_sem - 1] = 1.0
        weight = r.forward(st, [cam], features=mask)[0]["feat"][-1]
        st["sem"][who, n_sem - 1] = float("nan")
        feat = r.forward(st, [cam], features=mask)[0]["feat"]
        assert 0 < int((weight > 0).sum()) < weight.numel()
        assert torch.equal(torch.isnan(feat[-1]), weight > 0)
        assert torch.isfinite(feat[:-1]).all()


@pytest.mark.parametrize("mask,n_sem", [(abi.FEAT_RHO, 0), (abi.FEAT_SEM, 24), (7, 28), (7, 32)])
@pytest.mark.parametrize("cfg", [(8, 8, 1), (16, 8, 1), (32, 32, 4)])
def test_channel_blocks_of_every_width_agree(cfg, mask, n_sem):
    """The channel passes' two and four pixels per lane (the view alone and
    repeated; 32 and 36 channels keep two in the forward, 36 in both): the
    same images bit for bit, gradients that add up (the tolerance above)."""
    scene = synth.make_plain_scene(seed=4, n=300, sh_degree=1, log_scale_mean=-2.3)
    st = R.scene_to_device(scene)
    if n_sem:
        st["sem"] = torch.tensor(synth.make_semantics(300, n_sem), device="cuda")
    cam = synth.plain_camera(97, 61, t=0.4, bg=(0.2, 0.1, 0.3))
    r = R.Renderer(tile=cfg[:2], pixels_per_thread=cfg[2])
    one, many = R.Frame(), R.Frame()
    ref = r.forward(st, [cam], frame=one, features=mask)[0]
    d = _weights(cam, True)
    g = torch.Generator(device="cuda")
    g.manual_seed(8)
    d["feat"] = torch.randn(*ref["feat"].shape, generator=g, device="cuda")
    g1 = r.backward(st, [cam], one, [d])
    cams = _views(cam, cfg)
    outs = r.forward(st, cams, frame=many, features=mask)
    gn = r.backward(st, cams, many, [d] * len(cams))
    for v in (0, len(cams) // 2, len(cams) - 1):
        for k in ("rgb", "depth", "alpha", "feat"):
            assert torch.equal(outs[v][k], ref[k]), (v, k)
    for k in [*R.PARAM_NAMES] + (["sem"] if n_sem else []):
        want = g1[k].double() * len(cams)
        assert torch.linalg.norm(want) > 0, k
        assert torch.linalg.norm(gn[k].double() - want) <= 1e-4 * torch.linalg.norm(want), k
