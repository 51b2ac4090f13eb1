"""Rules of the device code that hold for every input and that no run can show:
checked on the source."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _code():
    for f in sorted(glob.glob(os.path.join(ROOT, "paper_2601_11338_gb300", "csrc", "*.cu*"))):
        yield os.path.basename(f), open(f).read()


def test_cluster_barriers_do_not_need_converged_warps():
    """barrier.cluster with .aligned is undefined where a warp's lanes may be
    apart, as they may after a branch on the lane."""
    for name, txt in _code():
        hits = re.findall(r"barrier\.cluster\.\w+[\w.:]*", txt)
        assert not [h for h in hits if "aligned" in h], name
