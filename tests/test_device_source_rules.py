"""Rules of the device code that no run shows reliably, checked on its source."""

import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2506_10911_b200", "csrc")


def code(path):
    with open(path) as f:
        text = f.read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def test_nothing_is_read_through_the_non_coherent_path():
    """Kernels here become resident while their predecessor in the stream still writes what they will read
    after their wait.  ld.global.nc, __ldg and const __restrict__ parameters all promise that the memory stays
    unwritten for as long as the kernel runs."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = code(path)
        assert "__ldg" not in text, path
        assert "ld.global.nc" not in text, path
        assert not re.search(r"\bconst\s+\w+\s*\*\s*__restrict__", text), path
