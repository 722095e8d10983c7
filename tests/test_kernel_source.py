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


@pytest.mark.parametrize("name", sorted(k for k, v in KERNELS.items() if "tcgen05.dealloc" in v[1]))
def test_a_kernel_that_gave_up_waits_for_its_copies(name):
    """A kernel with bounded waits leaves only when what it has in flight has had time to land: tensor copies and products
    are written into shared and tensor memory that is the next block's once this one has gone."""
    body = KERNELS[name][1]
    tail = body[:body.index("tcgen05.dealloc")]
    assert re.search(r"\(\*\(volatile int \*\)&ctl->abort_flag\)\s*__nanosleep\(\d{6,}\)"
                     r"|gave_up = \*\(volatile int \*\)&ctl->abort_flag != 0;.*if \(gave_up\)\s*__nanosleep\(\d{6,}\)", tail, re.S)


def test_the_one_launch_pass_stays_in_bounds_after_a_wait_that_ran_out():
    """The selection runs even when the CTA gave up a wait (its warps need not agree on that, and they share barriers),
    with whatever scores and counts it then finds: the places it stores at are brought into range, whatever they are."""
    body = KERNELS["evict_fused"][1]
    assert "int t = min(max((before & 0xffff) + min(eb, need_eq), 0), P.nkeep)" in body
    assert body.count("list[t] = ") == 2 and "for (int t = tid; t < P.nkeep; t += kFT) list[t] = t;" in body
    assert body.count("min(max(list[t0r + i") == 2     # and so are the positions that rows are read at


@pytest.mark.parametrize("name", ["decode_step", "gather_rows"])
def test_what_the_kernel_before_may_still_write_is_not_read_as_read_only(name):
    """These two read what the kernel right before them in the stream has written (the pruned cache, the kept positions) and
    may be set up while it runs: their inputs do not go through the read-only path, which is for data that nobody writes
    during a kernel's life."""
    params, body = KERNELS[name]
    assert "cudaGridDependencySynchronize" in body
    assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", params) and "__ldg" not in body
    with open(os.path.join(CSRC, {"decode_step": "jq_decode.cu", "gather_rows": "jq_gather.cu"}[name])) as f:
        assert "ld.global.nc" not in f.read()
