"""The autotuner times every tile shape that the library supports once: the
pixels per thread of a configuration reach no kernel, so a second candidate of
a shape would time the same kernels again.  No GPU."""
import os
import re

from paper_2311_18561_gb300 import build
from paper_2311_18561_gb300 import tune as T


def test_one_candidate_per_supported_tile_shape():
    text = open(os.path.join(build.SRC, "raster_common.cuh")).read()
    table = text[text.index("#define PVG_TILE_CONFIGS"):]
    supported = {tuple(int(v) for v in m) for m in re.findall(r"X\((\d+), (\d+), (\d+)\)", table)}
    assert len(supported) == 13
    assert set(T.CONFIGS) <= supported
    shapes = [c[:2] for c in T.CONFIGS]
    assert len(shapes) == len(set(shapes))
    assert set(shapes) == {c[:2] for c in supported}
