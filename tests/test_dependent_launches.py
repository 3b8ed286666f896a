"""Host checks of the launches behind one another (csrc/pdl.cuh)."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1609_01490_gb300", "csrc")


def test_no_read_only_loads_behind_a_producer():
    """Files whose kernels are launched behind another use no load that takes its data
    as constant for the whole kernel: the first kernel may still be writing it."""
    files = [f for f in glob.glob(os.path.join(CSRC, "*.cu")) if "launch_behind" in open(f).read()]
    assert len(files) >= 4
    for f in files:
        code = re.sub(r"//[^\n]*", "", open(f).read())
        assert not re.search(r"__ldg\s*\(|ld\.global\.nc", code), f
