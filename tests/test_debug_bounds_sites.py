"""The debug-bounds build checks every computed index: each read of the words' largest depths
(Window::zmax in csrc/fused.cu) follows a range check in the same statement."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_15183_gb300", "csrc")


def test_largest_depths_are_read_behind_a_range_check():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "fused.cu")).read())
    statements = [s for s in re.split(r"[;{}]", src) if "zmax[" in s and not re.search(r"zmax\[[^\]]*\]\s*=[^=]", s)]
    assert len(statements) == 2
    for s in statements:
        assert "YORO_BOUND(" in s[:s.index("zmax[")], s.strip()
