"""Launch choices take the device's multiprocessor count from the device: none
of a GB300's (152, or products of it with blocks per multiprocessor) stands in
the kernels' launch code as a number."""
import glob
import os
import re

from paper_1506_03745_gb300 import build


def test_no_multiprocessor_count_in_the_sources():
    found = []
    for path in glob.glob(os.path.join(build.CSRC, "*.cu*")):
        for n, line in enumerate(open(path), 1):
            code = line.split("//")[0]
            found += [(os.path.basename(path), n, k) for k in re.findall(r"\b(\d+)\b", code) if k in ("152", "1216", "2432")]
    assert not found, found
