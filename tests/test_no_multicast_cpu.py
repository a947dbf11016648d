"""No kernel copies into another CTA's shared memory: every rank of a multi-rank run executes
the same kernels, and none of them may use a TMA load with cluster multicast there.  (What a
commit of MMAs signals to the barriers of a CTA pair is no copy.)"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2506_07430_gb300", "csrc")


def test_no_multicast_copies():
    sources = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert sources
    for path in sources:
        for asm in re.findall(r"asm volatile\(.*?\);", open(path).read(), re.S):
            assert not ("cp.async" in asm and "multicast" in asm), (path, asm)
