"""The register-resident kernel's warps reach the group barrier at different places of the
program (a warp without a node waits in a loop of its own).  __syncthreads is defined in
conditional code only where the whole block takes the same branch, so the barrier there
has to be the one that counts threads."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1803_01215_gb300", "csrc",
                   "warp_solver.cuh")


def test_group_barrier_counts_its_threads():
    src = open(SRC).read()
    body = re.search(r"void group_sync\(\) \{(.*?)\n\}", src, re.S).group(1)
    assert "__syncthreads" not in body
    assert re.search(r"bar\.sync 1, %0;.*32 \* G", body)
    # the two branches on warp_on hold no other barrier
    for branch in re.findall(r"if \(warp_on\) \{(.*?)\n    \} else \{(.*?)\n    \}", src, re.S):
        assert all("__syncthreads" not in b for b in branch)
