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


def test_the_state_is_written_before_a_successor_may_start():
    """A caller's kernel launched by programmatic serialization may read weights ahead of its wait, and does start as
    soon as the kernel ahead of it lets it: so the outer step never does, and the other kernels that can end a call
    do so behind their own wait only (what went before them may have written weights)."""
    outer = code(os.path.join(CSRC, "nolo_outer.cu"))
    steps, mean = outer[:outer.index("group_mean_kernel(")], outer[outer.index("group_mean_kernel("):]
    assert "let_successor_start" not in steps
    for text in (mean, code(os.path.join(CSRC, "nolo_route.cu"))):
        lines = [ln.strip() for ln in text.splitlines() if ln.strip()]
        calls = [i for i, ln in enumerate(lines) if "let_successor_start" in ln]
        assert calls and all(lines[i - 1] == "wait_for_predecessors();" for i in calls)
