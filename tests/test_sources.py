"""The kernels' sources: what a library that every rank of a multi-GPU program loads must not hold."""
import glob
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1203_2394_gb300", "csrc")


def test_no_cluster_multicast():
    # a bulk load or a commit with cluster multicast is for programs of one GPU alone; libdpf.so is
    # one library for all, so no kernel of it may name one
    hits = [os.path.basename(p) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))
            if ".multicast::cluster" in open(p).read()]
    assert hits == []
