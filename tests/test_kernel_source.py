"""Rules that the kernels keep and that no run can be trusted to show broken, read off their source."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_10798_b200", "csrc")


def kernels():
    """name -> (parameter list, body) of every __global__ function."""
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\(((?:[^()]|\([^()]*\))*)\)\s*\{", text):
            if m.group(1) == "__launch_bounds__":
                continue
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            out[m.group(1)] = (m.group(2), text[m.end():i - 1])
    return out


KERNELS = kernels()
REMOTE = re.compile(r"map_shared_rank|peer_addr\(|push_f32\(")   # the ways into another CTA's shared memory


@pytest.mark.parametrize("name", sorted(k for k, v in KERNELS.items() if REMOTE.search(v[1])))
def test_a_cluster_has_started_before_its_shared_memory_is_touched(name):
    """Another CTA's shared memory may be accessed once that CTA runs: an arrival before the kernel waits for the one
    before it, and the wait ahead of the first access."""
    body = KERNELS[name][1]
    arrive, dep = body.find("barrier.cluster.arrive"), body.find("cudaGridDependencySynchronize")
    assert 0 <= arrive < dep
    wait = body.find("barrier.cluster.wait")
    assert dep < wait < REMOTE.search(body).start()


def test_the_cluster_kernels_are_found():
    assert {k for k, v in KERNELS.items() if REMOTE.search(v[1])} == {"decode_step", "evict_fused", "select_cluster"}
