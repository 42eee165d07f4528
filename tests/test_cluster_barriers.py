"""Kernels that read another CTA's shared memory: every access lies between a
cluster barrier that shows all CTAs of the cluster to be running and one that
keeps their shared memory until it has been read."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2404_06926_gb300", "csrc")


@pytest.mark.parametrize("name", ["gl_loss.cu", "gl_params.cu"])
def test_remote_shared_memory_lies_between_barriers(name):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    # a kernel's accesses follow the cluster_group it declares
    bodies = src.split("this_cluster()")[1:]
    assert bodies and all("map_shared_rank" in b for b in bodies)
    for body in bodies:
        syncs = [m.start() for m in re.finditer(r"cluster\.sync\(\)", body)]
        maps = [m.start() for m in re.finditer(r"map_shared_rank\(", body)]
        assert len(syncs) >= 2 and syncs[0] < maps[0] and maps[-1] < syncs[-1]
