"""The library is also what every rank of a multi-GPU (replica) run loads, so
no TMA load in its sources multicasts to a cluster (tcgen05.commit's arrival on
a pair's two barriers is no load)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_00835_gb300", "csrc")


def test_no_multicast_tma_load():
    files = glob.glob(os.path.join(CSRC, "*.cu*"))
    assert files
    for f in files:
        with open(f) as fh:
            text = fh.read()
        for stmt in re.findall(r"asm volatile\((.*?)\);", text, re.S):
            joined = "".join(re.findall(r'"([^"]*)"', stmt))
            if "cp.async.bulk" in joined:
                assert "multicast" not in joined, os.path.basename(f)
