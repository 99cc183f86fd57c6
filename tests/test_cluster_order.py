"""Another CTA's shared memory may be touched only once that CTA is known to run: in every
kernel that does so a cluster barrier has been waited for first.  Read off the sources, since
a run shows nothing as long as the CTAs of a cluster happen to start together."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_22983_gb300", "csrc")


def _bodies(text):
    """(name, body) of every __global__ function."""
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\([^{;]*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_cluster_barrier_before_remote_memory(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    remote = [(k, b) for k, b in _bodies(text) if "map_shared_rank" in b]
    if name in ("lv_kernels.cu", "lv_sched.cu"):
        assert remote
    for kernel, body in remote:
        before = body[:body.index("map_shared_rank")]
        assert "cluster.sync()" in before or "barrier.cluster.wait" in before, kernel
