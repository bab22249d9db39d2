"""Copies that a cluster's CTAs share by TMA multicast belong to programs of one GPU only; the
library also runs as one replica per GPU, so its sources hold none."""
import glob
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_multicast_in_the_sources():
    for path in glob.glob(os.path.join(ROOT, "paper_1409_0297_gb300", "csrc", "*")):
        with open(path) as f:
            assert "multicast" not in f.read(), path
