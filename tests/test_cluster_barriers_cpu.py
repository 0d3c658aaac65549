"""Source check: cluster barriers that follow divergent code must not be the `.aligned` forms, which want all threads of a warp
at the instruction together (undefined otherwise, and a stuck cluster cannot be provoked in a test)."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_aligned_cluster_barriers():
    found = 0
    for path in glob.glob(os.path.join(ROOT, "paper_2208_00763_b200", "csrc", "*.cu*")):
        for form in re.findall(r'"barrier\.cluster\.[a-z.]+', open(path).read()):
            found += 1
            assert "aligned" not in form, "%s: %s" % (path, form)
    assert found == 2
