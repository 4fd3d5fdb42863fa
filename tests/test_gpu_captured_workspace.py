"""A captured graph holds the buffers of its renderer's workspace, so with a
fixed pair capacity none of them may move when frames of another size follow:
frames of at most 8,192 items, whose pair expansion works in shorter chunks,
allocate nothing on a workspace that a larger frame has filled (the allocation
hook would fail them), leave a graph captured before them valid and can be
captured themselves.
"""
import pytest
import torch

from paper_2311_18561_gb300 import abi
from paper_2311_18561_gb300 import render as R
from paper_2311_18561_gb300 import synth

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(autouse=True)
def _clear_hook():
    yield
    abi.lib().pvg_debug_fail_allocations(0)


@pytest.mark.parametrize("tile", [(8, 8), (16, 16)])
@pytest.mark.parametrize("capacity", [1 << 20, 1 << 22])
def test_small_frames_leave_the_workspace_where_it_is(capacity, tile):
    cam = synth.plain_camera(640, 480, t=0.4)
    big = R.scene_to_device(synth.make_plain_scene(seed=3, n=9000, log_scale_mean=-5.0))
    small = R.scene_to_device(synth.make_plain_scene(seed=4, n=2000, log_scale_mean=-4.0))
    want_small = R.Renderer(tile=tile).forward(small, [cam])[0]["rgb"].clone()
    r = R.Renderer(tile=tile, sync_sizes=False, pair_capacity=capacity)
    held, other = R.Frame(), R.Frame()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        outs = r.forward(big, [cam], frame=held)
        r.forward(big, [cam], frame=other)
        small_outs = r.alloc_images([cam])
    stream.synchronize()
    assert held.stats()[2] == 0  # within the capacity
    want = outs[0]["rgb"].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        r.forward(big, [cam], outs=outs, frame=held)
    abi.lib().pvg_debug_fail_allocations(1)
    with torch.cuda.stream(stream):
        r.forward(small, [cam], outs=small_outs, frame=other)
    abi.lib().pvg_debug_fail_allocations(0)
    stream.synchronize()
    assert other.stats()[2] == 0 and torch.equal(small_outs[0]["rgb"], want_small)
    outs[0]["rgb"].zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(outs[0]["rgb"], want)


@pytest.mark.parametrize("capacity", [1 << 20, 1 << 22])
def test_a_small_frame_can_be_captured_after_a_larger_one(capacity):
    cam = synth.plain_camera(640, 480, t=0.4)
    big = R.scene_to_device(synth.make_plain_scene(seed=3, n=9000, log_scale_mean=-5.0))
    small = R.scene_to_device(synth.make_plain_scene(seed=4, n=2000, log_scale_mean=-4.0))
    want = R.Renderer(tile=(8, 8)).forward(small, [cam])[0]["rgb"].clone()
    r = R.Renderer(tile=(8, 8), sync_sizes=False, pair_capacity=capacity)
    frame, stream = R.Frame(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        outs = r.forward(big, [cam], frame=frame)
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        r.forward(small, [cam], outs=outs, frame=frame)
    graph.replay()
    torch.cuda.synchronize()
    assert frame.stats()[2] == 0 and torch.equal(outs[0]["rgb"], want)
