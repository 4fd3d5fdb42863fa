"""Distributed shared memory may be accessed only once every CTA of the
cluster is known to have started, which only a barrier of the cluster shows:
in every function of the CUDA sources a cluster barrier is waited for before
the first address of another CTA's shared memory is formed, and another one
after the last (no CTA leaves while another reads or writes its memory).
Read from the sources, since the missing wait is a race that a run need not
show.  No GPU."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2311_18561_gb300", "csrc")
WAIT = re.compile(r"\b(?:this_cluster\(\)|cluster)\s*\.\s*(?:sync|barrier_wait)\s*\(")
REMOTE = re.compile(r"\bmap_shared_rank\s*\(|\bmapa\b")


def _functions(text):
    """(name, body) of the functions at namespace scope."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    text = re.sub(r"__(?:cluster_dims|launch_bounds)__\s*\((?:[^()]|\([^()]*\))*\)", "", text)
    for m in re.finditer(r"\b(\w+)\s*\([^;{}]*\)\s*(?:const\s*)?\{", text):
        depth, i = 1, m.end()
        while depth and i < len(text):
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


def test_remote_shared_memory_lies_between_cluster_barriers():
    seen = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for name, body in _functions(open(path).read()):
            remote = [m.start() for m in REMOTE.finditer(body)]
            if not remote or name in ("if", "constexpr", "for", "while"):
                continue
            waits = [m.start() for m in WAIT.finditer(body)]
            where = "%s: %s" % (os.path.basename(path), name)
            assert waits and waits[0] < remote[0], where + ": accessed before the cluster's CTAs are known to run"
            assert waits[-1] > remote[-1], where + ": a CTA may leave while its memory is accessed"
            seen.append(name)
    assert {"tile_order", "k_rgb_loss_finish"} <= set(seen)
