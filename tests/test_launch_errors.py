"""Every kernel launch in the library has its error read before the next kernel of the call is launched: a launch that failed must not be
followed by kernels that read what it would have written."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_15211_b200", "csrc")
FILES = sorted(f for f in glob.glob(os.path.join(CSRC, "*.cu")) if "<<<" in open(f).read())


@pytest.mark.parametrize("path", FILES, ids=[os.path.basename(f) for f in FILES])
def test_launch_errors_are_read(path):
    text = open(path).read()
    for m in re.finditer("<<<", text):
        # up to the next timed scope, dependent launch or end of the function
        end = min(i for i in (text.find(s, m.end()) for s in ("prof_begin(", "launch_dependent(", "\n}")) if i >= 0)
        assert "cudaGetLastError()" in text[m.end():end], f"line {text.count(chr(10), 0, m.start()) + 1}: the launch's error is not read before what follows"
