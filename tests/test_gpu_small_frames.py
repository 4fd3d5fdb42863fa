"""Frames of at most 8,192 items take one CTA per sorting stage.  The same
scene with Gaussians behind the camera appended, so that it takes the general
stages, gives the same lists and images bit for bit: around the edges of the
CTA's shares, with few and many pairs, for one view and several, with and
without the pair count read back, and beyond the pair capacity.
"""
import numpy as np
import pytest
import torch

from paper_2311_18561_gb300 import render as R
from paper_2311_18561_gb300 import synth

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

SMALL_ITEMS = 8192


def _scenes(n, n_views, log_scale):
    """(scene, the same with invisible Gaussians behind it): device tensors."""
    s = synth.make_plain_scene(seed=n, n=n, log_scale_mean=log_scale)
    extra = synth.make_plain_scene(seed=1, n=SMALL_ITEMS // n_views + 1)
    extra["mu"][:, 2] -= 100.0  # behind the camera at z = -4
    extra["vel"][:] = 0.0
    both = {k: np.concatenate([s[k], extra[k]]) for k in R.PARAM_NAMES}
    return R.scene_to_device(s), R.scene_to_device(both)


def _render(st, cams, tile, sync, capacity, n, stride):
    r = R.Renderer(tile=tile[:2], pixels_per_thread=tile[2], sync_sizes=sync, pair_capacity=capacity)
    fr = R.Frame()
    outs = r.forward(st, cams, frame=fr)
    torch.cuda.synchronize()
    tx, ty = R.tiles_of(cams[0], tile[:2])
    ex = fr.export(tx * ty * len(cams))
    gid = ex["sorted_gid"].astype(np.int64)
    ex["sorted_gid"] = gid // stride * n + gid % stride  # the small scene's ids
    return outs, ex, fr.stats()


@pytest.mark.parametrize("sync", [True, False])
@pytest.mark.parametrize("n,n_views,tile,log_scale", [
    (1, 1, (16, 16, 1), -2.0), (33, 1, (8, 8, 1), -2.0), (1023, 1, (16, 16, 1), -4.0), (1024, 2, (16, 8, 1), -4.0),
    (1025, 1, (32, 32, 4), -3.0), (2000, 1, (16, 16, 1), -3.0), (2000, 4, (8, 8, 1), -2.0),
    (8192, 1, (16, 16, 1), -4.0), (8192, 1, (8, 8, 2), -2.5)])
def test_small_frames_match_the_general_stages(n, n_views, tile, log_scale, sync):
    st, big = _scenes(n, n_views, log_scale)
    cams = [synth.plain_camera(161, 119, t=0.3 + 0.1 * v) for v in range(n_views)]
    capacity = 1 << 22
    a, ea, sa = _render(st, cams, tile, sync, capacity, n, n)
    b, eb, sb = _render(big, cams, tile, sync, capacity, n, n + SMALL_ITEMS // n_views + 1)
    assert sa == sb and sa[2] == 0
    if not sync and 0 < sa[1] <= SMALL_ITEMS:  # a capacity that the one-CTA tile sort takes too
        a, ea, sc = _render(st, cams, tile, sync, SMALL_ITEMS, n, n)
        assert sc == sa
    for k in ea:
        np.testing.assert_array_equal(ea[k], eb[k], err_msg=k)
    for x, y in zip(a, b):
        for k in ("rgb", "depth", "alpha"):
            assert torch.equal(x[k], y[k]), k


@pytest.mark.parametrize("capacity", [100, 4000, 20000])
def test_small_frame_beyond_its_pair_capacity_reports_it(capacity):
    st, big = _scenes(4000, 1, -2.0)
    cam = [synth.plain_camera(161, 119)]
    _, ea, sa = _render(st, cam, (16, 16, 1), False, capacity, 4000, 4000)
    _, eb, sb = _render(big, cam, (16, 16, 1), False, capacity, 4000, 4000 + SMALL_ITEMS + 1)
    assert sa == sb and sa[1] > capacity and sa[2] != 0
    np.testing.assert_array_equal(ea["pair_vals"][:capacity], eb["pair_vals"][:capacity])
    np.testing.assert_array_equal(ea["ranges"], eb["ranges"])


def test_differentiable_renders_share_frames_only_behind_one_another():
    """Gradients of interleaved differentiable renders (two pending at once,
    on two streams, and one dropped without a backward pass) equal those of
    renders on their own; a second backward pass of one render is refused."""
    st = R.scene_to_device(synth.make_plain_scene(seed=2, n=500))
    cams = [synth.plain_camera(64, 48, t=t) for t in (0.3, 0.5, 0.7)]
    r = R.Renderer()

    def start(cam):
        p = {k: v.clone().requires_grad_(True) for k, v in st.items()}
        return p, R.render_differentiable(p, cam, r)

    def finish(p, out, retain=False):
        g = torch.autograd.grad(out, list(p.values()), [torch.ones_like(o) for o in out], retain_graph=retain)
        torch.cuda.synchronize()
        return g

    want = [finish(*start(c)) for c in cams]
    assert len(r._frames) == 1
    pending = [start(c) for c in cams[:2]]
    start(cams[2])  # dropped: its frame goes back
    got = [finish(*p) for p in pending]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        got.append(finish(*start(cams[2])))
    for a, b in zip(want, got):
        for x, y in zip(a, b):
            assert torch.linalg.norm(x - y) <= 1e-5 * torch.linalg.norm(x)
    assert len(r._frames) <= 4
    assert {s for s, _ in r._frames} == {torch.cuda.current_stream().cuda_stream, side.cuda_stream}
    p, out = start(cams[0])
    finish(p, out, retain=True)
    with pytest.raises(Exception):
        finish(p, out)
    r.close()
    assert not r._frames
