"""No arrival on another CTA's mbarrier carries a cluster-scope release (CPU).
Such a release waits for the thread's global stores: in the gate-up epilogue,
which arrives once a tile, that made calls of little K up to 1.5 times as
slow (8000 tokens, hidden 64, inter 6912: 73.7 us, 47.8 without)."""
import glob
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_15171_gb300", "csrc")


def test_remote_arrivals_do_not_wait_for_stores():
    text = ""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path, encoding="utf-8") as f:
            text += f.read()
    assert "mbarrier.arrive.shared::cluster" in text
    assert "mbarrier.arrive.release.cluster" not in text
