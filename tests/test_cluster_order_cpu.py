"""Memory order of the cluster kernels (csrc/cluster.cuh, the users of its
barriers): what one CTA reads of another's shared memory is ordered before the
other's next writes there by the cluster barrier alone, so every arrival has to
release and every wait to acquire.  A relaxed arrival after a gather gives no
such order, whatever depends on the gathered values."""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_15797_gb300", "csrc")


def _sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            yield os.path.basename(path), f.read()


def test_every_cluster_arrival_releases_and_every_wait_acquires():
    arrivals = waits = 0
    for name, text in _sources():
        for op in re.findall(r"barrier\.cluster\.arrive[.\w]*", text):
            assert op == "barrier.cluster.arrive.release", (name, op)
            arrivals += 1
        for op in re.findall(r"barrier\.cluster\.wait[.\w]*", text):
            assert op == "barrier.cluster.wait.acquire", (name, op)
            waits += 1
    assert arrivals and waits
