"""Distributed shared memory may be written only once every CTA of the cluster
has started, which a cluster barrier shows and the launch of a cluster does not.
In every kernel that maps an address of another CTA, a wait on the cluster
barrier stands before the first mapped address."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1705_05783_gb300", "csrc")
REMOTE = re.compile(r"\bmap_rank\(|\bcl_store\(|\bmap_shared_rank\(|\bmapa\.")
BARRIER = re.compile(r"\bcluster_sync\(\)|\bcluster_wait\(\)|\bcl_sync\(\)|\bcl\.sync\(\)|\bcl\.barrier_wait\(")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__", src):
            depth, start = 0, None
            for i in range(m.end(), len(src)):
                if src[i] == "{":
                    start = i if depth == 0 else start
                    depth += 1
                elif src[i] == "}":
                    depth -= 1
                    if depth == 0:
                        break
                elif src[i] == ";" and depth == 0:
                    break
            if start is None:
                continue
            names = re.findall(r"(\w+)\s*\(", src[m.end():start])
            name = next(n for n in names if n.startswith("k_"))
            yield f"{os.path.basename(path)}:{name}", src[start:i + 1]


REACH = [(name, body) for name, body in _kernels() if REMOTE.search(body)]


def test_the_cluster_kernels_are_found():
    assert {n.split(":")[1] for n, _ in REACH} >= {"k_sweep", "k_residual_small", "k_coarse_solve_cluster",
                                                   "k_coarse_solve_twisted"}


@pytest.mark.parametrize("name, body", REACH, ids=[n for n, _ in REACH])
def test_a_cluster_barrier_comes_before_remote_shared_memory(name, body):
    first = BARRIER.search(body)
    assert first, "no cluster barrier"
    assert first.start() < REMOTE.search(body).start()
