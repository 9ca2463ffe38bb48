"""Distributed shared memory may be accessed only while the other block runs, which a cluster
barrier establishes: in every kernel that maps a peer's shared memory, one completes before the
first access and one follows the last.  Checked in the source, since the hardware usually starts a
cluster's blocks together and a missing barrier need not show; no GPU needed."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2301_09662_gb300", "csrc")
REMOTE = re.compile(r"map_shared_rank|\bmapa\b|ld\.shared::cluster|st\.(async\.)?shared::cluster")
BARRIER = re.compile(r"\.sync\(\)|barrier_wait\(\)|barrier\.cluster\.wait")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__", code):
            start = code.index("{", m.start())
            depth, end = 0, start
            for end in range(start, len(code)):
                depth += {"{": 1, "}": -1}.get(code[end], 0)
                if depth == 0:
                    break
            body = code[start:end]
            if REMOTE.search(body):
                yield pytest.param(body, id=re.search(r"(\w+)\s*\(const", code[m.start():start]).group(1))


@pytest.mark.parametrize("body", list(_kernels()))
def test_cluster_barrier_around_remote_accesses(body):
    at = [m.start() for m in REMOTE.finditer(body)]
    assert BARRIER.search(body, 0, at[0]), "a peer's shared memory is accessed before any cluster barrier"
    assert BARRIER.search(body, at[-1]), "a block may leave while a peer still accesses its shared memory"
