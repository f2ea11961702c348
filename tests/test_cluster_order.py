"""Order of cluster barriers and accesses to another CTA's shared memory, from the kernels'
source (a missing barrier shows as a rare lost value at best, so it is not looked for by
running): a CTA may touch a peer's shared memory only once the peer is known to have started,
and a CTA may exit only once no peer touches its own any more."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_09231_gb300", "csrc")
REMOTE = r"\b(st_cluster\d|mbar_arrive_remote|tma_load_2d_pair|mma_bf16_pair|mma_commit_pair)\("
BARRIER = r"\b(cluster_sync_all|cluster_wait)\("


def kernels():
    """(name, body without comments) of every kernel that accesses another CTA's shared memory."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+_kernel)\(", src):
            i = src.index("{", m.end())
            depth, j = 1, i + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[j], 0)
                j += 1
            if re.search(REMOTE, src[i:j]):
                yield m.group(1), src[i:j]


def test_the_cluster_kernels_are_found():
    assert {n for n, _ in kernels()} == {"attn_tc_kernel", "gemm_pair_kernel", "gemm_splitk_kernel",
                                         "rel_l1_cluster_kernel"}


@pytest.mark.parametrize("name,body", list(kernels()), ids=lambda v: v if v.endswith("_kernel") else "")
def test_remote_accesses_lie_between_cluster_barriers(name, body):
    remote = [m.start() for m in re.finditer(REMOTE, body)]
    barriers = [m.start() for m in re.finditer(BARRIER, body)]
    assert barriers and barriers[0] < remote[0], f"{name}: a remote access before the first cluster barrier"
    assert barriers[-1] > remote[-1], f"{name}: no cluster barrier after the last remote access"
    # a split barrier is waited on as often as it is arrived at
    assert len(re.findall(r"\bcluster_arrive\(", body)) == len(re.findall(r"\bcluster_wait\(", body))
