"""Order of cluster barriers and distributed shared memory in the kernel sources.

A CTA may touch the shared memory of another CTA of its cluster only while that CTA is known to
run: a barrier of the whole cluster stands before the kernel's first such access and after its
last one."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1607_05816_gb300", "csrc")
BARRIER = re.compile(r"\bunit_sync<kCl>\(\)|\bcl(?:uster)?\.sync\(\)|this_cluster\(\)\.sync\(\)|barrier\.cluster\.wait")
KERNELS = ["alg1_cluster", "batch_solve", "grid_pass_tc3"]
REMOTE = re.compile(r"\bmap_shared_rank\(")


def kernels():
    """(file, name, body without comments) of every __global__ function that maps remote shared memory."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for at in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^{;]*?\)\s+)?(\w+)\s*\(", src):
            i = src.find("{", at.end())
            j, depth = i, 0
            while True:
                depth += {"{": 1, "}": -1}.get(src[j], 0)
                j += 1
                if depth == 0:
                    break
            if REMOTE.search(src[i:j]):
                out.append((os.path.basename(path), at.group(1), src[i:j]))
    return out


def test_kernels_are_found():
    assert {name for _, name, _ in kernels()} == set(KERNELS)


@pytest.mark.parametrize("name", KERNELS)
def test_remote_shared_memory_between_cluster_barriers(name):
    body = next(b for _, n, b in kernels() if n == name)
    barriers = [m.start() for m in BARRIER.finditer(body)]
    remote = [m.start() for m in REMOTE.finditer(body)]
    assert barriers[0] < remote[0], "no cluster barrier before the first access to another CTA's shared memory"
    assert barriers[-1] > remote[-1], "no cluster barrier after the last access to another CTA's shared memory"
