"""Kernels launched in clusters, read as text: shared memory of another CTA may be touched only while that CTA is known to run.  In
every kernel that stores into it, arrives on its barriers or signals them, a cluster barrier is waited for in front of the first such
access and behind the last."""
import os
import re

import pytest

import paper_2512_05746_b200

CSRC = os.path.join(os.path.dirname(paper_2512_05746_b200.__file__), "csrc")
REMOTE = re.compile(r"st\.shared::cluster|st_async_v4\(|mbar_arrive_cluster\(|mma_commit_to\(|mma_commit_pair\(|tma_load_\dd_pair\(")
BARRIER = re.compile(r"cluster_sync_all\(|cluster_wait\(")


def kernels():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name), encoding="utf-8") as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__[^;{]*?\b(\w+kernel)\s*\([^;{]*\)\s*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            body = text[m.end(): end]
            if REMOTE.search(body):
                yield pytest.param(body, id=m.group(1))


@pytest.mark.parametrize("body", list(kernels()))
def test_other_ctas_are_known_to_run_while_their_shared_memory_is_touched(body):
    touched = [m.start() for m in REMOTE.finditer(body)]
    waited = [m.start() for m in BARRIER.finditer(body)]
    assert waited and waited[0] < touched[0] and touched[-1] < waited[-1]
