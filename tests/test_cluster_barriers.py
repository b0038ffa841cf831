"""Kernels that reach into the shared memory of their cluster's other CTAs: a
CTA may only be reached once it is known to have started and as long as it
cannot have left, so a barrier of the whole cluster comes before the first
such access and another one after the last.  A missing barrier seldom shows in
a run (a cluster's CTAs mostly start together), so the source is read."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
REACH = r"map_shared_rank|mapa\.|shared::cluster"
BARRIER = r"cluster\.sync\(\)|barrier\.cluster\.wait"


def _cluster_kernels():
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2205_03251_gb300", "csrc", "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__cluster_dims__", src):
            start = src.index("{", src.index(") {", m.start()))
            depth, end = 0, start
            for end in range(start, len(src)):
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                if depth == 0:
                    break
            yield os.path.basename(path), src[start:end]


def test_cluster_kernels_wait_before_and_after_they_reach_other_ctas():
    kernels = list(_cluster_kernels())
    assert kernels
    for name, body in kernels:
        reach = [m.start() for m in re.finditer(REACH, body)]
        waits = [m.start() for m in re.finditer(BARRIER, body)]
        if not reach:
            continue
        assert waits and waits[0] < reach[0], f"{name}: reaches another CTA before all have started"
        assert waits[-1] > reach[-1], f"{name}: a CTA may leave while another reaches it"
