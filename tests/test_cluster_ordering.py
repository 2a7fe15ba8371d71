"""Every cluster barrier of the device code orders memory.  A colour pass of the cluster cycle reads old values
of its own colour and then overwrites them in the shared memory of all CTAs of the cluster; in the PTX memory
model only an arrival with release and a wait with acquire order those reads before the remote writes
(a relaxed arrival orders nothing, whatever the timing).  Checked on the source: the race itself shows in no
result that a test could wait for."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_13046_gb300", "csrc")


def test_cluster_barriers_are_release_acquire():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"barrier\.cluster\.(arrive|wait)([.\w]*)", text):
            want = ".release" if m.group(1) == "arrive" else ".acquire"
            assert want in m.group(2), (os.path.basename(path), m.group(0))
            seen += 1
    assert seen
