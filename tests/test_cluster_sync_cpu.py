"""Cluster kernels, by their source (CPU only): a CTA may touch the shared memory
of another one only after a cluster barrier has shown that it runs."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_02798_gb300", "csrc")
REMOTE = re.compile(r"map_shared_rank|mbar_arrive_cluster|mma_commit_pair|peer_addr")
BARRIER = re.compile(r"cluster_sync\(|\.sync\(\)|\.barrier_wait\(")


def kernels():
    """(file, name, body) of every __global__ function."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__\s+void", src):
            at = src.index("{", m.end())
            while src[at - 1] == "=":
                at = src.index("{", at + 1)
            name = re.findall(r"(\w+)\s*\(", re.sub(r"__\w+__\s*\([^)]*\)", "", src[m.end():at]))[0]
            depth, end = 0, at
            while True:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
                if depth == 0:
                    break
            yield f, name, src[at:end]


REMOTE_KERNELS = [k for k in kernels() if REMOTE.search(k[2])]


def test_the_cluster_kernels_are_found():
    assert {"cg_vec_kernel", "rownorm_tc3_kernel", "rownorm_tc2_kernel"} <= {k[1] for k in REMOTE_KERNELS}


@pytest.mark.parametrize("f,name,body", REMOTE_KERNELS, ids=[k[1] for k in REMOTE_KERNELS])
def test_a_cluster_barrier_comes_before_the_first_remote_access(f, name, body):
    barrier = BARRIER.search(body)
    assert barrier and barrier.start() < REMOTE.search(body).start(), f"{f}: {name}"
