"""Rules of the particle passes that no run can show, read off their sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_00935_gb300", "csrc")


def test_no_pass_reads_through_the_read_only_path():
    """A pass may be resident while the pass before it writes the grid that it will gather, so it may not
    read through the non-coherent path, which is defined for memory that nothing writes meanwhile."""
    for name in ("mpm_kernels.cuh", "mpm_common.cuh", "controller.cu"):
        with open(os.path.join(CSRC, name)) as f:
            code = re.sub(r"//[^\n]*", "", f.read())
        assert not re.search(r"__ldg\s*\(|ld\.global(\.\w+)*\.nc", code), name
