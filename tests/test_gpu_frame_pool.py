"""The idle frames that a renderer keeps for render_differentiable: bounded,
the least recently used one dropped first, given up when memory runs out,
never lent to a stream that only has the handle of a destroyed one, kept past
the stream that used them, and never left to a captured backward pass.
"""
import ctypes

import pytest
import torch

from paper_2311_18561_gb300 import abi
from paper_2311_18561_gb300 import render as R
from paper_2311_18561_gb300 import synth

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

CAM = synth.plain_camera(64, 48, t=0.3)


@pytest.fixture(autouse=True)
def _clear_hook():
    yield
    abi.lib().pvg_debug_fail_allocations(0)


@pytest.fixture(scope="module")
def scene():
    return R.scene_to_device(synth.make_plain_scene(seed=2, n=500))


def _forward(st, r, cam=CAM):
    p = {k: v.clone().requires_grad_(True) for k, v in st.items()}
    return p, R.render_differentiable(p, cam, r)


def _backward(p, out, **kw):
    return torch.autograd.grad(out, list(p.values()), [torch.ones_like(o) for o in out], **kw)


def _step(st, r):
    g = _backward(*_forward(st, r))
    torch.cuda.synchronize()
    return g


def test_the_least_recently_used_frame_is_dropped(scene):
    r = R.Renderer()
    streams = [torch.cuda.Stream() for _ in range(R._FrameLease.KEEP + 1)]
    torch.cuda.synchronize()
    for s in streams:
        with torch.cuda.stream(s):
            _step(scene, r)
    kept = [f for _, f in r._frames]
    assert len(kept) == R._FrameLease.KEEP
    with torch.cuda.stream(streams[-1]):
        assert R._FrameLease(r).frame is kept[-1]  # the last stream's own
    with torch.cuda.stream(streams[0]):
        assert R._FrameLease(r).frame not in kept  # dropped for it
    r.close()
    assert not r._frames


def test_idle_frames_are_given_up_when_memory_runs_out(scene):
    other = R.scene_to_device(synth.make_plain_scene(seed=3, n=20_000))
    want = R.Renderer().forward(other, [CAM])[0]["rgb"].clone()
    r = R.Renderer()
    _step(scene, r)
    assert len(r._frames) == 1
    abi.lib().pvg_debug_fail_allocations(1)
    out = r.forward(other, [CAM])[0]["rgb"]
    torch.cuda.synchronize()
    assert torch.equal(out, want) and not r._frames
    # without idle frames the failure is the caller's
    plain = R.Renderer()
    abi.lib().pvg_debug_fail_allocations(1)
    with pytest.raises(abi.PVGError) as e:
        plain.forward(other, [CAM])
    assert e.value.status == 2
    # an idle frame gone, the backward pass that needs the memory runs too
    abi.lib().pvg_debug_fail_allocations(0)
    _step(scene, r)
    p, out = _forward(scene, r)  # takes the idle frame
    q, out2 = _forward(scene, r)
    _backward(q, out2)           # leaves another
    fr = R.Frame()
    r.forward(other, [CAM], frame=fr)
    abi.lib().pvg_debug_fail_allocations(1)
    g = r.backward(other, [CAM], fr, [dict(rgb=torch.ones(3, 48, 64, device="cuda"))])
    torch.cuda.synchronize()
    assert torch.isfinite(g["mu"]).all() and not r._frames
    _step(scene, r)
    r.free_idle_frames()
    assert not r._frames
    _backward(p, out)


def _external_stream():
    """(handle, destroy): a stream of the caller's own."""
    rt = torch.cuda.cudart()
    s = ctypes.c_void_p()
    assert int(rt.cudaStreamCreate(ctypes.addressof(s))) == 0
    return s.value, lambda: rt.cudaStreamDestroy(s.value)


def test_a_destroyed_streams_handle_does_not_lend_its_frames(scene):
    """Whether a new stream gets a destroyed one's handle is CUDA's own
    choice, so the idle frame is entered under a new stream's handle."""
    r = R.Renderer()
    handle, destroy = _external_stream()
    with torch.cuda.stream(torch.cuda.ExternalStream(handle)):
        _step(scene, r)
        (idle,) = [f for _, f in r._frames]
        lease = R._FrameLease(r)
        assert lease.frame is idle  # the same stream
        lease.release()
    torch.cuda.synchronize()
    destroy()
    made = [_external_stream() for _ in range(8)]
    try:
        ids = {idle.stream_key[1]} | {R._stream_key(torch.cuda.ExternalStream(h))[1] for h, _ in made}
        assert 0 not in ids and len(ids) == len(made) + 1
        new = made[0][0]
        with torch.cuda.stream(torch.cuda.ExternalStream(new)):
            r._frames[:] = [(new, idle)]
            idle.stream_key = (new, idle.stream_key[1])
            assert R._FrameLease(r).frame is not idle
    finally:
        torch.cuda.synchronize()
        r.close()
        for _, d in made:
            d()


def test_frames_outlive_the_stream_that_used_them(scene):
    cam2 = synth.plain_camera(48, 32)
    r, fr = R.Renderer(), R.Frame()
    handle, destroy = _external_stream()
    with torch.cuda.stream(torch.cuda.ExternalStream(handle)):
        _step(scene, r)
        r.forward(scene, [cam2], frame=fr)
    torch.cuda.synchronize()
    assert len(r._frames) == 1
    destroy()
    fr.close()
    r.close()


def test_a_captured_backward_pass_is_refused(scene):
    """A graph would keep using a frame that other renders are lent."""
    r = R.Renderer(sync_sizes=False, pair_capacity=1 << 20)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        want = _step(scene, r)
        p, out = _forward(scene, r)
        seeds = [torch.ones_like(o) for o in out]
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with pytest.raises(abi.PVGError) as e:
        with torch.cuda.graph(graph, stream=stream):
            torch.autograd.grad(out, list(p.values()), seeds, retain_graph=True)
    assert e.value.status == 1 and not r._frames
    with torch.cuda.stream(stream):  # the render can still be differentiated
        got = torch.autograd.grad(out, list(p.values()), seeds)
    torch.cuda.synchronize()
    for a, b in zip(want, got):
        assert torch.linalg.norm(a - b) <= 1e-5 * torch.linalg.norm(a)
    r.close()
