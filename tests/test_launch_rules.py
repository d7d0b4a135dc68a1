"""Read from the sources, comments aside.  Rules that choose a kernel or its grid
count the SMs of the device at hand, not those of one device (152, and their
multiples 304, 608).  Cluster barriers are not of the .aligned form, which is
undefined where a warp's lanes may arrive apart."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_11790_gb300", "csrc")


def test_no_device_sm_count_in_the_code():
    bad = []
    for path in glob.glob(os.path.join(CSRC, "*")):
        code = re.sub(r"/\*.*?\*/|//[^\n]*|\"(?:\\.|[^\"\\])*\"", "", open(path).read(), flags=re.S)
        bad += [f"{os.path.basename(path)}: {m}" for m in re.findall(r"(?<![\w.])(?:148|152|303|304|608)\b", code)]
    assert not bad, bad


def test_no_aligned_cluster_barrier():
    for path in glob.glob(os.path.join(CSRC, "*")):
        code = re.sub(r"/\*.*?\*/|//[^\n]*", "", open(path).read(), flags=re.S)
        assert not re.search(r"barrier\.cluster\.[a-z.]*aligned", code), os.path.basename(path)
