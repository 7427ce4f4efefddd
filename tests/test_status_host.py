"""The device status word (first word of every workspace)."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2608_21308_b200" / "csrc"


def test_no_kernel_clears_the_status_word():
    """A kernel's blocks run in no particular order: one that cleared the word could erase what a wait that gave up had written.  The word
    is cleared in stream order before a launch; kernels only set it, from zero."""
    for f in sorted(CSRC.glob("*.cu*")):
        for line in f.read_text().splitlines():
            assert not re.search(r"\*\s*(a|wc|t)\.status\s*=(?!=)", line), f"{f.name}: {line.strip()}"
