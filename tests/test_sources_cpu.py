"""Rules of the CUDA sources that no run would show to be broken."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_03588_b200", "csrc")


def test_no_read_only_loads():
    """The kernels may start while the kernel that writes their inputs still runs, so nothing may be read by the loads
    that are for data unchanged over a kernel's whole life (they are not ordered by the wait for that kernel)."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"__ldg\b|ld\.global(\.\w+)*\.nc|__restrict__", code), path
