"""Every tensor-map load of the kernels writes the shared memory of the CTA that issues it: the library also serves runs
with a rank per GPU, where loads that write several CTAs of a cluster at once are not to be used."""
import glob
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_07401_gb300", "csrc")


def test_no_load_writes_several_ctas():
    files = sorted(glob.glob(os.path.join(CSRC, "*")))
    found = [os.path.basename(f) for f in files if "multicast" in open(f).read()]
    assert files and not found
