"""Two CTAs that share a tile's products hand over accumulator sums through
mbarriers: the release and the acquire must both be at cluster scope, or the
PTX memory model orders nothing between the CTAs.  A wrong scope gives wrong
results only by a rare timing on the GPU, so the source is checked."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KERNEL = os.path.join(ROOT, "paper_2609_04663_gb300", "csrc", "prodsum_f64w_kernel.cuh")


def _body(text, name):
    m = re.search(r"%s\([^)]*\)\n\{\n(.*?)\n\}\n" % name, text, re.S)
    return m.group(1)


def test_duo_barriers_release_and_acquire_at_cluster_scope():
    text = open(KERNEL).read()
    signal, wait = _body(text, "void signal_duo"), _body(text, "bool wait_duo")
    assert "mbarrier.arrive.release.cluster." in signal
    assert "mbarrier.try_wait.parity.acquire.cluster." in wait and "mbar_wait(" not in wait
    # every wait of a duo's barrier goes through wait_duo
    assert not re.search(r"mbar_(try_)?wait\(duo_", text)
    assert len(re.findall(r"wait_duo\(duo_(first|done)", text)) == 3
