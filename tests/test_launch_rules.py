"""Launch shapes follow the device's SM count as the context has it: no kernel source
builds one part's count (152 of a GB300, or a share of it) into its rules."""
import glob
import os
import re

from test_cluster_start import CSRC, strip_comments


def test_no_sm_count_is_built_in():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = strip_comments(open(path).read())
        found = re.findall(r"(?<![\w.])(?:152|151|148|304|76|38)(?![\w.])", code)
        assert found == [], (os.path.basename(path), found)
