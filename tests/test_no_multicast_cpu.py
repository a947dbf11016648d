"""No kernel copies into another CTA's shared memory: every rank of a multi-rank run executes
the same kernels, and none of them may use a TMA load with cluster multicast there."""
import glob
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2506_07430_gb300", "csrc")


def test_no_cluster_multicast():
    sources = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert sources
    for path in sources:
        assert "multicast" not in open(path).read(), path
