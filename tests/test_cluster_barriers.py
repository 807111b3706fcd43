"""CPU: kernels that write into the shared memory of other CTAs of their cluster do so only between
two cluster barriers: one before the first remote access (a peer may not have started before it)
and one after the last (a peer may have left).  Read from the sources: an access outside them can
fault the GPU, so that no run shows it."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1705_01893_gb300", "csrc")


def _kernels():
    """(file:name, body without comments) of every __global__ function that maps remote addresses."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^{;]*?\)\s*)?(\w+)\([^)]*\)\s*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            body = text[m.end():end - 1]
            if "map_shared_rank" in body or "mapa." in body:
                yield f"{os.path.basename(path)}:{m.group(1)}", body


KERNELS = dict(_kernels())


def test_kernels_found():
    assert "mm_small.cu:k_small" in KERNELS


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_remote_accesses_lie_between_cluster_barriers(name):
    """The barriers of the entry and the exit stand in the kernel's own block, outside any loop,
    branch or lambda."""
    body = KERNELS[name]
    remote = [m.start() for m in re.finditer(r"map_shared_rank|mapa\.", body)]
    top = []                                  # barriers at the kernel's own nesting depth
    for m in re.finditer(r"\bcl\.sync\(\)", body):
        head = body[:m.start()]
        if head.count("{") == head.count("}"):
            top.append(m.start())
    assert top and min(top) < min(remote), "no cluster barrier before the first remote access"
    assert max(top) > max(remote), "no cluster barrier after the last remote access"
