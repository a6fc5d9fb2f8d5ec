"""The build recompiles when a header changes: every file that the CUDA sources
include by name is among those whose age it compares."""
import glob
import os
import re

from paper_1901_05118_gb300 import build


def test_every_included_header_is_watched():
    watched = {os.path.basename(p) for p in build.header_files()}
    named = set()
    for path in glob.glob(os.path.join(build.CSRC, "*")):
        with open(path) as f:
            named.update(re.findall(r'^#include "([^"]+)"', f.read(), re.M))
    assert named and named <= watched
