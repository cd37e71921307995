"""The order of a cluster's barriers and its CTAs' accesses to one another's
shared memory, read from the kernels' sources on CPU: CUDA requires that a CTA
is known to have started before a peer touches its shared memory, so in every
kernel a barrier of the cluster comes before the first such access. (Nothing
but an unlucky schedule shows a missing one at run time.)"""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2609_08368_gb300", "csrc")
PEER = re.compile(r"\b(st_dsmem_f64|ld_dsmem_f4|st_async_f4)\s*\(")
BARRIER = re.compile(r"\b(cluster_sync_all|cluster_wait)\s*\(")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", src):
            start = src.index("{", m.end())
            depth, end = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
            yield m.group(1), src[start:end]


BODIES = dict(_kernels())
PEERED = sorted(n for n, b in BODIES.items() if PEER.search(b))


def test_the_kernels_are_found():
    assert {"k_adv_grpo", "k_bwd", "k_short"} <= set(BODIES)
    assert PEERED == ["k_stats", "k_stream", "k_sweep"]


@pytest.mark.parametrize("name", PEERED)
def test_a_barrier_comes_before_the_first_access_to_a_peer(name):
    first = BARRIER.search(BODIES[name])
    assert first and first.start() < PEER.search(BODIES[name]).start()
