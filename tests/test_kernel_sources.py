"""Rules of the kernel sources that no result shows (no GPU needed)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_20357_gb300", "csrc")


def _code(path):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)


def test_no_kernel_reads_through_the_non_coherent_path():
    """Every kernel may start before its predecessor has ended, so its inputs are not read-only for its lifetime, which
    is what non-coherent loads require."""
    files = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))
    assert files
    for path in files:
        assert not re.findall(r"\b__ldg\b|\b__restrict__\b|ld\.global\.nc", _code(path)), os.path.basename(path)
