"""Rules of the persistent kernels that can be checked without a GPU."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2303_17679_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def test_cluster_barrier_takes_diverged_warps():
    """barrier.cluster.*.aligned is undefined for a warp whose lanes have not
    rejoined; the phases of the kernels end in loops of per-lane trip counts."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        for ins in re.findall(r'"(barrier\.cluster\.[a-z.]+)', open(path).read()):
            assert ".aligned" not in ins, (os.path.basename(path), ins)
    assert "barrier.cluster.wait.acquire" in source("gridsync.cuh")
