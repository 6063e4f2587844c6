"""What host code keeps about a GPU is kept for each device: a kernel's raised
shared-memory limit or an SM count in a plain static variable would be the first
device's on every other one.  Read from the sources (the machines these tests
run on have at most one GPU)."""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1901_07499_gb300", "csrc")


def test_static_variables_are_indexed_by_device():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as fh:
            text = re.sub(r"//[^\n]*", "", fh.read())
        for m in re.finditer(r"^\s+static (?:bool|int|unsigned|size_t|cudaError_t|void\*) (\w+)((?:\[\w+\])*)\s*[=;]",
                             text, re.M):
            found.append((os.path.basename(path), m.group(1), m.group(2)))
    assert len(found) >= 5
    assert [f for f in found if not f[2].endswith("[64]")] == []
