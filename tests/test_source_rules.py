"""Properties of the CUDA sources that one GPU cannot show."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_1907_06821_gb300", "csrc", "*.cu*")))


def test_kernel_attributes_are_not_behind_a_flag_of_the_process():
    """A kernel's shared-memory limit belongs to the kernel on one device.  Set once per process, on
    the device of the first call, it leaves the launches of a context on another device to fail."""
    assert len(SOURCES) > 10
    for path in SOURCES:
        text = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"std::(once_flag|call_once)", text), path
        assert not re.search(r"\bstatic\s+(bool|int)\s+\w+\s*=", text), path
