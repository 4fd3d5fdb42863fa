"""The work counts of a frame (pvg_frame_eval_count) equal those of a plain
float64 walk over the exported lists and records, for every tile shape, at
ragged sizes, for one view and several, with pixels that stop early.

Tolerance: a count differs where an alpha or a transmittance lies within the
float32 rounding of its threshold (a few 1e-6 relative), which fewer than one
in 10,000 of these entries does; a pixel whose stop moves by one entry adds at
most its list's few entries.  1e-3 of the totals.
"""
import numpy as np
import pytest
import torch

from paper_2311_18561_gb300 import render as R
from paper_2311_18561_gb300 import synth

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def _counts(ex, cams, tile):
    """(E, blended) by walking every pixel's list."""
    evals = blends = 0
    first = 0
    for cam in cams:
        tx, ty = R.tiles_of(cam, tile)
        for t in range(tx * ty):
            lo, hi = ex["ranges"][first + t]
            rec = ex["records"][ex["pair_vals"][lo:hi]].astype(np.float64)
            px, py = np.meshgrid(np.arange(tile[0]) + t % tx * tile[0], np.arange(tile[1]) + t // tx * tile[1])
            inside = (px < cam["width"]) & (py < cam["height"])
            px, py = px[inside] + 0.5, py[inside] + 0.5
            trans, going = np.ones(px.size), np.ones(px.size, bool)
            for u, v, a, b, c, o, _, hx, _, _, _, hy in rec:
                dx, dy = px - u, py - v
                evals += int((going & (np.abs(dx) <= hx) & (np.abs(dy) <= hy)).sum())
                alpha = o * np.exp(-0.5 * (a * dx * dx + 2 * b * dx * dy + c * dy * dy))
                on = going & (alpha >= 1 / 255)
                blends += int(on.sum())
                after = trans * (1 - np.minimum(alpha, 0.99))
                going &= ~(on & (after < 1e-4))
                trans = np.where(on & going, after, trans)
        first += tx * ty
    return evals, blends


@pytest.mark.parametrize("n_views", [1, 2])
@pytest.mark.parametrize("tile", [(8, 8, 1), (16, 8, 1), (32, 8, 1), (16, 16, 1), (32, 16, 1), (32, 32, 4), (16, 32, 4)])
def test_counts_match_a_walk_over_the_lists(tile, n_views):
    scene = synth.make_plain_scene(seed=6, n=400, log_scale_mean=-2.3)
    scene["opacity"][::3] = 1.0  # pixels stop early
    st = R.scene_to_device(scene)
    cams = [synth.plain_camera(75 + 6 * v, 53, t=0.3 + 0.2 * v) for v in range(n_views)]
    r, fr = R.Renderer(tile=tile[:2], pixels_per_thread=tile[2]), R.Frame()
    r.forward(st, cams, frame=fr)
    got = R.eval_count(r, fr)
    tiles = sum(int(np.prod(R.tiles_of(c, tile[:2]))) for c in cams)
    want = _counts(fr.export(tiles), cams, tile[:2])
    assert want[1] > 0 and want[0] >= want[1]
    for g, w in zip(got, want):
        assert abs(g - w) <= 1e-3 * w, (got, want)
