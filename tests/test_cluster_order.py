"""Kernels that touch another block's shared memory wait for the cluster's blocks first.

Distributed shared memory may be accessed only once every block of the cluster has started, which
a cluster barrier ahead of the first access guarantees. A kernel without one mostly works, so the
order is read from the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2604_21095_gb300", "csrc")
REMOTE = r"st\.shared::cluster|st_cluster_u32\s*\(|mbar_arrive_cluster\s*\(|tma_load_2d_pair\s*\("
BARRIER = r"cluster_sync_all\s*\(|cluster_wait\s*\("


def _kernels():
    """(file, kernel name, body without comments) of every kernel."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        with open(os.path.join(CSRC, f)) as fh:
            src = re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", fh.read()), flags=re.S)
        for m in re.finditer(r"__global__", src):
            open_at = src.index("{", m.end())
            name = re.findall(r"(k_\w+)\s*\(", src[m.end():open_at])[0]
            depth, end = 0, open_at
            for end in range(open_at, len(src)):
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                if depth == 0:
                    break
            yield f, name, src[open_at:end]


REMOTE_KERNELS = [k for k in _kernels() if re.search(REMOTE, k[2])]


def test_the_known_kernels_are_found():
    assert {"k_hit_stats", "k_tc2_scan"} <= {k[1] for k in REMOTE_KERNELS}


@pytest.mark.parametrize("f,name,body", REMOTE_KERNELS, ids=[k[1] for k in REMOTE_KERNELS])
def test_cluster_barrier_comes_before_the_first_remote_access(f, name, body):
    barrier = re.search(BARRIER, body)
    assert barrier, f"{name} ({f}) touches other blocks' shared memory without a cluster barrier"
    assert barrier.start() < re.search(REMOTE, body).start(), (f, name)
