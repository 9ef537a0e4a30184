"""Distributed shared memory may be touched only once every CTA of the cluster has
started: a kernel that writes another CTA's shared memory passes a cluster barrier
before its first such write. Read from the sources (a write that comes too early is
undefined, so it is not run)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1911_10630_gb300", "csrc")
BARRIER = re.compile(r"\b(cl\.sync|team_sync)\s*\(")
# writes through a mapped address, and the helpers that write to all CTAs
REMOTE = re.compile(r"\*\s*cl\.map_shared_rank\s*\(|st\.(async\.)?shared::cluster|\b(team_sum|cluster_sum\w*|cluster_max)\s*<")


def _kernels():
    """(file, name, body) of every kernel."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\((?:[^()]|\([^()]*\))*\) )?(\w+)\s*\(", src):
            at = src.index("{", m.end())
            depth, end = 0, at
            while True:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
                if depth == 0:
                    break
            yield os.path.basename(path), m.group(1), src[at:end]


CLUSTER = [(f, n, b) for f, n, b in _kernels() if REMOTE.search(b)]


def test_the_cluster_kernels_are_found():
    assert {n for _, n, _ in CLUSTER} >= {"cg64_kernel", "cluster_pair_kernel", "cluster_mg_kernel"}


@pytest.mark.parametrize("file,name,body", CLUSTER, ids=[n for _, n, _ in CLUSTER])
def test_a_barrier_comes_before_the_first_remote_write(file, name, body):
    first = REMOTE.search(body).start()
    barrier = BARRIER.search(body)
    assert barrier and barrier.start() < first, f"{file}: {name}"
