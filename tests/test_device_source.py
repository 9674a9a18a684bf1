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


def test_training_reads_what_it_writes_after_the_wait():
    """The two kernels of a training step follow one another as dependent
    launches: before its wait a kernel may read the samples only, not the
    parameters, moments, operands or sums that the launches write."""
    text = _source("mlp.cu")
    for kernel, written in (("k_mlp_train_samples(TrainArgs a)", ("a.W", "a.ops")),
                            ("k_mlp_train_update(UpdateArgs a)", ("a.theta", "a.m[", "a.v[", "a.acc", "a.ops", "a.W"))):
        body = text[text.index(kernel):]
        body = body[:body.index("\n}\n")]
        waits = [body.find(w) for w in ("wait_previous()", "after_previous()") if w in body]
        assert waits and min(waits) > 0
        for name in written:
            assert name in body and body.index(name) > min(waits), (kernel, name)
