"""Cluster barriers are executed by whole warps.

The .aligned forms of barrier.cluster are undefined where the lanes of a warp do not execute
them together (a CTA may leave while others still read its shared memory, or none may ever
leave), and nothing brings lanes together again after a ragged loop or an early return.  A GPU
run shows neither, so this reads the sources: every such instruction has a __syncwarp() right
before it, in the one header that all kernels take it from."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1903_05133_gb300", "csrc")


def _sources():
    paths = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))
    assert paths
    return {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read()) for p in paths}


def test_cluster_barrier_instructions_have_one_home():
    for name, text in _sources().items():
        if name != "ptx.cuh":
            assert "barrier.cluster" not in text, name


def test_warps_converge_before_every_aligned_cluster_barrier():
    text = _sources()["ptx.cuh"]
    statements = [s.strip() for s in re.split(r"[;{}](?=\s)", text) if s.strip()]
    found = 0
    for before, s in zip(statements, statements[1:]):
        if "barrier.cluster" not in s:
            continue
        found += 1
        assert s.count("barrier.cluster") == 1 and before == "__syncwarp()", s
    assert found == text.count("barrier.cluster") > 0
