"""Rules of the device code whose breach is undefined behaviour, so that no run
on a GPU could be relied on to show it: they are checked on the source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2301_10674_gb300", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_cluster_barrier_takes_divergent_warps():
    """The warps of the DEM cluster kernel reach the barrier with lane groups
    that ran loops of different lengths; the .aligned forms need all lanes of a
    warp at the instruction together."""
    forms = re.findall(r"barrier\.cluster\.[a-z.]+", _source("particles.cu"))
    assert sorted(forms) == ["barrier.cluster.arrive.release", "barrier.cluster.wait.acquire"]
