"""Kernels that store into the shared memory of their cluster's other CTAs: a barrier of the whole cluster has to come
before the first such store (every CTA must have started) and after the last one (none may have left).  Read from the
sources: a kernel without them is undefined, not wrong every time."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_17742_gb300", "csrc")


def _kernels():
    """(name, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\([^;{]*\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            yield m.group(1), text[m.end():i]


def test_cluster_barrier_around_remote_stores():
    seen = 0
    for name, body in _kernels():
        puts = [m.start() for m in re.finditer(r"\bput_cluster\s*\(", body)]
        if not puts:
            continue
        seen += 1
        syncs = [m.start() for m in re.finditer(r"\bcluster_sync\s*\(\s*\)", body)]
        assert syncs and syncs[0] < puts[0], f"{name}: stores into the cluster before its first barrier"
        assert syncs[-1] > puts[-1], f"{name}: no barrier after the last store"
        # both barriers outside every loop: at the body's own depth
        for at in (syncs[0], syncs[-1]):
            assert body[:at].count("{") == body[:at].count("}"), name
    assert seen >= 1
