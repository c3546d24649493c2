"""The library's kernels run on every rank of a multi-GPU job, so none of them may load with TMA multicast: each CTA
issues its own loads."""
import glob
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_tma_multicast_in_the_sources():
    files = [f for d in ("paper_1909_08596_gb300/csrc", "include", "synth/csrc")
             for f in glob.glob(os.path.join(ROOT, d, "*")) if os.path.isfile(f)]
    assert any(f.endswith("rns.cu") for f in files)
    assert not [f for f in files if ".multicast::cluster" in open(f).read()]
